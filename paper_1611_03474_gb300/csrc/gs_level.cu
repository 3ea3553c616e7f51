// gs_level.cu -- one level of the adaptive partition (section 2.2):
//   * the coefficient tensor A of every examined cube (eqs polynew,
//     tensor1, tensor2): per atom the Legendre projection of its 1-D
//     Gaussian factor on each axis (eqs poly2_1..3, n = 3) with the C0
//     endpoint correction (eqs poly3, condition1, alpha), weighted by
//     exp(D r^2) and accumulated as a rank-one update;
//   * the estimate of [L, U] by the two-level truncated SVD (eqs matrix1,
//     SVD1-SVD7, Sxyz, bound1-bound3) and the decision
//     discard / accept / split (steps 1-3 of section 2.2).
//
// Layout: cubes are examined in octets (the 8 children of one split parent,
// or a 2x2x2 block of root cubes).  One warp accumulates one octet: lane
// (child c = lane/4, j = lane%4) owns the 16 entries A_c[j][*][*].  The 8
// children share the candidate atoms (cell rows around the parent box) and,
// per atom and axis, two child intervals, so each atom's coefficients are
// computed once per octet and used by up to 8 cubes.  Estimation runs one
// thread per cube.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>

#include "gs_host.cuh"

// ---------------------------------------------------------------- quadrature
// Gauss-Legendre nodes t_k and folded weights W_kj = (2j+1)/2 * w_k * L_j(t_k),
// so that alpha_j = sum_k W_kj f(t_k) for j = 0, 1 (the end points give the
// other two).  Variants with 8, 16 and 24 nodes.
#define GQ_VARIANTS 3
#define GQ_MAX 24
__constant__ double c_gq_t[GQ_VARIANTS][GQ_MAX];
__constant__ double c_gq_W[GQ_VARIANTS][GQ_MAX][2];
__constant__ float c_gq_tf[GQ_VARIANTS][GQ_MAX];
__constant__ float c_gq_Wf[GQ_VARIANTS][GQ_MAX][2];
static const int kGqN[GQ_VARIANTS] = {8, 16, 24};

// nodes of P_n as eigen-free Newton iteration in long double, started from
// Tricomi's asymptotic estimate
static void gl_rule(int n, long double *t, long double *w)
{
    const long double pi = 3.141592653589793238462643383279502884L;
    for (int k = 1; k <= n; k++) {
        long double th = pi * (4.0L * k - 1.0L) / (4.0L * n + 2.0L);
        long double x = (1.0L - (n - 1.0L) / (8.0L * n * n * n)) * cosl(th);
        long double dp = 0;
        for (int it = 0; it < 60; it++) {
            long double pm1 = 1.0L, p = x;
            for (int m = 2; m <= n; m++) {
                long double pn = ((2.0L * m - 1.0L) * x * p - (m - 1.0L) * pm1) / m;
                pm1 = p;
                p = pn;
            }
            dp = n * (pm1 - x * p) / (1.0L - x * x);
            long double dx = p / dp;
            x -= dx;
            if (fabsl(dx) < 1e-19L) break;
        }
        t[k - 1] = x;
        w[k - 1] = 2.0L / ((1.0L - x * x) * dp * dp);
    }
}

// Re-expansion of a cubic Legendre series on a half interval: for the lower
// (h = 0) or upper (h = 1) half of [-1,1], R[h][p][j] = (2p+1)/2 times the
// integral of L_j((t + sigma)/2) L_p(t) over [-1,1] (sigma = -1 or +1), so
// that the child's coefficients are R times the parent's.
__constant__ double c_reexp[2][4][4];

static bool g_gq_ready[64];

int gs_quadrature_init(void)
{
    int dev = 0;
    GS_CHECK(cudaGetDevice(&dev));
    if (dev >= 0 && dev < 64 && g_gq_ready[dev]) return GS_OK;
    static double t[GQ_VARIANTS][GQ_MAX], W[GQ_VARIANTS][GQ_MAX][2];
    static float tf[GQ_VARIANTS][GQ_MAX], Wf[GQ_VARIANTS][GQ_MAX][2];
    for (int v = 0; v < GQ_VARIANTS; v++) {
        long double tt[GQ_MAX], ww[GQ_MAX];
        int n = kGqN[v];
        gl_rule(n, tt, ww);
        for (int k = 0; k < GQ_MAX; k++) {
            long double x = k < n ? tt[k] : 0.0L, wk = k < n ? ww[k] : 0.0L;
            long double L[2] = {1.0L, x};
            t[v][k] = (double)x;
            tf[v][k] = (float)x;
            for (int j = 0; j < 2; j++) {
                W[v][k][j] = (double)((2.0L * j + 1.0L) / 2.0L * wk * L[j]);
                Wf[v][k][j] = (float)W[v][k][j];
            }
        }
    }
    {
        // 4-point Gauss-Legendre integrates the degree-6 products exactly
        long double t4[4], w4[4];
        gl_rule(4, t4, w4);
        auto L = [](int j, long double x) -> long double {
            switch (j) {
            case 0: return 1.0L;
            case 1: return x;
            case 2: return (3.0L * x * x - 1.0L) / 2.0L;
            default: return (5.0L * x * x * x - 3.0L * x) / 2.0L;
            }
        };
        static double R[2][4][4];
        for (int h = 0; h < 2; h++)
            for (int p = 0; p < 4; p++)
                for (int j = 0; j < 4; j++) {
                    long double acc = 0.0L, sg = h ? 1.0L : -1.0L;
                    for (int q = 0; q < 4; q++) acc += w4[q] * L(j, (t4[q] + sg) / 2.0L) * L(p, t4[q]);
                    R[h][p][j] = (double)((2.0L * p + 1.0L) / 2.0L * acc);
                }
        GS_CHECK(cudaMemcpyToSymbol(c_reexp, R, sizeof(R)));
    }
    GS_CHECK(cudaMemcpyToSymbol(c_gq_t, t, sizeof(t)));
    GS_CHECK(cudaMemcpyToSymbol(c_gq_W, W, sizeof(W)));
    GS_CHECK(cudaMemcpyToSymbol(c_gq_tf, tf, sizeof(tf)));
    GS_CHECK(cudaMemcpyToSymbol(c_gq_Wf, Wf, sizeof(Wf)));
    if (dev >= 0 && dev < 64) g_gq_ready[dev] = true;
    return GS_OK;
}

// ---------------------------------------------------------------- 1-D coefficients
// The four C0-corrected Legendre coefficients of exp(-D (x - xi)^2) on an
// interval of half-width hh whose centre lies m from the atom are
//   alpha_j = exp(-D m^2) Phi_j(beta),  beta = 2 D hh m,
// with Phi_j entire and depending on a^2 = D hh^2 alone (one level's
// constants).  For f(t) = exp(-beta t - a^2 t^2) on [-1, 1] the projection
// gives Phi_0 = 1/2 int f and Phi_1 = 3/2 int f t, and the endpoint
// correction turns the other two into (f(-1) + f(1))/2 - Phi_0 and
// (f(1) - f(-1))/2 - Phi_1.  Phi_0, Phi_2 are even and Phi_1, Phi_3 odd in
// beta; their power series converge for all beta.  A call needs one
// exponential and four short polynomials per interval, where the quadrature
// takes 5 to 24 exponentials and two more for the end points.  In a mesh of
// 20,000 atoms the FP64 accumulation, bound by the FP64 pipe, went from 88.2
// to 43.9 ms, the FP32 one (with the reordered updates below) from 2.38 to
// 2.05 ms; the tensors' errors against 64 bits are no larger (FP64: 1.2e-15
// of sum|A| at most, as before; FP32: 3.4e-7 of the term sizes, before 5.9e-7).
//
// series_coeffs: the polynomials in s = mu^2, mu = beta / B in [-1, 1] (odd
// ones times mu), B at least the largest |beta| of an atom that reaches the
// interval (within R of it).  The Taylor series, economised: from the highest
// power down, each term t_n s^n gives t_n 2^(1-2n) T*_n(s) away (T*_n the
// Chebyshev polynomial on [0, 1]), an error of at most |t_n| 2^(1-2n), until
// the sum of these would pass tol; the smallest K of Ks (ascending) that
// holds the rest is taken.  Returns K, or 0 when none does.  All differences
// are taken term by term, so nothing cancels.
#define SERIES_MAX 20
struct Series {
    double kappa;               // mu = kappa m
    double c[4][SERIES_MAX];
};
// B = 2^(e/8), on a fixed scale of eight steps per octave: inputs that differ
// a little in their largest radius share the polynomials
#define SERIES_NONE (1 << 20)
static int series_scale(double D, double hh, double R)
{
    const double bmax = 2.0 * D * hh * (R + hh);
    if (!(D * hh * hh <= 4.0) || !(bmax <= 14.0) || !(bmax > 1e-30)) return SERIES_NONE;
    return (int)ceil(8.0 * log2(bmax));
}
// exp(-D m^2) stays in gs_exp's range for |m| <= R + 3 hh
static bool series_range64(const GsProblem &P, double hh)
{
    return P.D * (P.pad + 3.0 * hh) * (P.pad + 3.0 * hh) <= 690.0;
}
// exp(-D m^2) stays above the flush range (2^-126) for every atom that
// reaches an interval
static bool series_range32(const GsProblem &P, double hh)
{
    return P.D * (P.pad + hh) * (P.pad + hh) <= 85.0;
}
int gs_coeff_class(const GsProblem &P, int level)
{
    const double hh = 0.5 * gs_h(P, level);
    return 4 * series_scale(P.D, hh, P.pad) + (series_range64(P, hh) ? 2 : 0) + (series_range32(P, hh) ? 1 : 0);
}
static int series_coeffs(double D, double hh, double R, double tol, const int *Ks, int nK, Series *out)
{
    constexpr int NT = 48;
    static const struct Table {
        double T[NT][NT];       // monomial coefficients of T*_n
        Table()
        {
            for (int n = 0; n < NT; n++)
                for (int i = 0; i < NT; i++) T[n][i] = 0.0;
            T[0][0] = 1.0;
            T[1][0] = -1.0;
            T[1][1] = 2.0;
            for (int n = 2; n < NT; n++)
                for (int i = 0; i <= n; i++)
                    T[n][i] = (i > 0 ? 4.0 * T[n - 1][i - 1] : 0.0) - 2.0 * T[n - 1][i] - T[n - 2][i];
        }
    } tab;
    const int scale = series_scale(D, hh, R);
    if (scale == SERIES_NONE) return 0;
    const double a2 = D * hh * hh, B = exp2(scale / 8.0), B2 = B * B;
    double t[4][NT];
    int N = 0;
    double f = 1.0;             // B^(2k) / (2k)!
    for (int k = 0; k < NT; k++) {
        double e0 = 0, e1 = 0, d0 = 0, d1 = 0, g = 1.0;   // g = (-a^2)^n / n!
        for (int n = 0; n < 60 && fabs(g) > 1e-20; n++) {
            const double u = 1.0 / (2 * k + 2 * n + 1), v = 3.0 / (2 * k + 2 * n + 3);
            e0 += g * u;
            e1 += g * v;
            d0 += g * (1.0 - u);
            d1 += g * (1.0 - v);
            g *= -a2 / (n + 1);
        }
        const double fo = f * B / (2 * k + 1);
        t[0][k] = f * e0;
        t[1][k] = -fo * e1;
        t[2][k] = f * d0;
        t[3][k] = -fo * d1;
        N = k + 1;
        if (k > 4 && f + fo < 1e-3 * tol) break;
        f *= B2 / ((2 * k + 1) * (2.0 * k + 2));
    }
    // give terms away until tol is reached
    double lost = 0.0;
    int need = N;
    for (; need > 1; need--) {
        const int n = need - 1;
        double d = 0.0;
        for (int q = 0; q < 4; q++) d = fmax(d, fabs(t[q][n]));
        d = ldexp(d, 1 - 2 * n);
        if (lost + d > tol) break;
        lost += d;
        for (int q = 0; q < 4; q++) {
            const double c = ldexp(t[q][n], 1 - 2 * n);
            for (int i = 0; i < n; i++) t[q][i] -= c * tab.T[n][i];
            t[q][n] = 0.0;
        }
    }
    int K = 0;
    for (int i = 0; i < nK && !K; i++)
        if (Ks[i] >= need) K = Ks[i];
    if (!K) return 0;
    for (int q = 0; q < 4; q++)
        for (int k = 0; k < K; k++) out->c[q][k] = k < N ? t[q][k] : 0.0;
    out->kappa = 2.0 * D * hh / B;
    return K;
}

// Node count of the quadrature, which serves what the series does not (wide
// intervals, very large D R^2): its error stays below ~1e-14 (FP64) or 2e-7
// of the Gaussian's peak (FP32) for sqrt(D)*hh up to each limit.
static int gq_variant(double D, double hh, bool fp32)
{
    const double a = sqrt(D) * hh;
    if (fp32) return a <= 1.0 ? 0 : 1;   // 8 or 16 nodes
    return a <= 0.25 ? 0 : (a <= 1.0 ? 1 : 2);   // 8, 16 or 24 nodes
}

// ---------------------------------------------------------------- octet geometry
struct Octet {
    int64_t I, J, K;   // parent coords (children at 2I+dx, ...)
    uint8_t vmask;     // valid children
};

__device__ __forceinline__ Octet octet_of(const GsProblem &P, int level, const uint64_t *parents,
                                          const uint8_t *vmask, int64_t o)
{
    Octet q;
    if (parents) {
        uint64_t k = parents[o];
        q.I = gk_x(k); q.J = gk_y(k); q.K = gk_z(k);
        q.vmask = vmask ? vmask[o] : 0xFF;
        if (level == 0) {
            // root blocks: drop children outside the root grid
            for (int c = 0; c < 8; c++) {
                int64_t x = 2 * q.I + (c & 1), y = 2 * q.J + ((c >> 1) & 1), z = 2 * q.K + (c >> 2);
                if (x >= P.nroot[0] || y >= P.nroot[1] || z >= P.nroot[2]) q.vmask &= (uint8_t)~(1u << c);
            }
        }
    } else {
        // root blocks of 2x2x2 cubes, x fastest
        int64_t bx = (P.nroot[0] + 1) / 2, by = (P.nroot[1] + 1) / 2;
        q.I = o % bx;
        q.J = (o / bx) % by;
        q.K = o / (bx * by);
        uint8_t m = 0;
        for (int c = 0; c < 8; c++) {
            int64_t x = 2 * q.I + (c & 1), y = 2 * q.J + ((c >> 1) & 1), z = 2 * q.K + (c >> 2);
            if (x < P.nroot[0] && y < P.nroot[1] && z < P.nroot[2]) m |= (uint8_t)(1u << c);
        }
        q.vmask = m;
    }
    return q;
}

// ---------------------------------------------------------------- FP64 accumulate
#define ACC_WARPS 4
#define ACC_Q 64

// one axis: C0-corrected Legendre coefficients of exp(-D (x - xi)^2) on
// [e0,e1] and [e1,e2] (the two child intervals), FP64; `need` selects the
// intervals (bit 0: [e0,e1], bit 1: [e1,e2]) some accumulated child uses
template <int GV, int NQ>
struct Quad64 {
    __device__ __forceinline__ void axis(double xi, double e0, double e1, double e2, double D,
                                         double *out /* [2][4] */, int need) const
    {
        double f0 = (need & 1) ? gs_exp(-D * (e0 - xi) * (e0 - xi)) : 0.0;
        double f1 = gs_exp(-D * (e1 - xi) * (e1 - xi));
        double f2 = (need & 2) ? gs_exp(-D * (e2 - xi) * (e2 - xi)) : 0.0;
#pragma unroll
        for (int h = 0; h < 2; h++) {
            if (!((need >> h) & 1)) continue;
            double lo = h ? e1 : e0, hi = h ? e2 : e1;
            double m = __dmul_rn(0.5, __dadd_rn(lo, hi)) - xi, hh = __dmul_rn(0.5, __dsub_rn(hi, lo));
            double a0 = 0, a1 = 0;
#pragma unroll
            for (int k = 0; k < NQ; k++) {
                double d = fma(hh, c_gq_t[GV][k], m);
                double f = gs_exp(-D * d * d);
                a0 = fma(c_gq_W[GV][k][0], f, a0);
                a1 = fma(c_gq_W[GV][k][1], f, a1);
            }
            double fa = h ? f1 : f0, fb = h ? f2 : f1;
            out[4 * h + 0] = a0;
            out[4 * h + 1] = a1;
            out[4 * h + 2] = 0.5 * (fa + fb) - a0;
            out[4 * h + 3] = 0.5 * (fb - fa) - a1;
        }
    }
};
template <int K>
struct Series64 {
    double kappa, c[4][K];
    __device__ __forceinline__ void axis(double xi, double e0, double e1, double e2, double D, double *out,
                                         int need) const
    {
#pragma unroll
        for (int h = 0; h < 2; h++) {
            if (!((need >> h) & 1)) continue;
            const double m = 0.5 * (h ? e1 + e2 : e0 + e1) - xi;
            const double mu = kappa * m, s = mu * mu, E = gs_exp(-D * m * m), o = mu * E;
            double p[4];
#pragma unroll
            for (int q = 0; q < 4; q++) {
                p[q] = c[q][K - 1];
#pragma unroll
                for (int k = K - 2; k >= 0; k--) p[q] = fma(p[q], s, c[q][k]);
                out[4 * h + q] = p[q] * ((q & 1) ? o : E);
            }
        }
    }
};

// split: warps that share an octet, 1 or ACC_WARPS.  With few octets (a recheck)
// one warp is alone on its SM quarter for an octet's hundreds of atoms: the
// block's warps then test every fourth 32 candidates each, compute the
// coefficients of 128 queued atoms at once and update a quarter of the
// entries (one k of the four) each.  Atoms are queued in candidate order and
// every entry adds them in that order in either form, so a cube's tensor
// does not depend on how many octets share its launch.
// BATCH: octet o belongs to molecule mol[o], whose problem is probs[mol[o]]
// (the molecules of one launch share D and the coefficient class, so one set
// of polynomials or one quadrature rule serves all)
template <class C, bool BATCH>
__global__ void __launch_bounds__(32 * ACC_WARPS) k_accum_f64(const __grid_constant__ GsProblem P0, int level,
                                                               const uint64_t *parents, const uint8_t *vmask,
                                                               int64_t n_oct, int split,
                                                               const __grid_constant__ C coef,
                                                               double *__restrict__ A_out,
                                                               unsigned long long *pairs,
                                                               const GsProblem *__restrict__ probs,
                                                               const int32_t *__restrict__ mol)
{
    // per queued atom: 3 axes x 2 intervals x 4 (x times w); a warp's part of
    // these belongs to its octet, or all of them to the block's
    __shared__ double s_cf[32 * ACC_WARPS][25];
    __shared__ int s_qi[ACC_Q * ACC_WARPS];
    __shared__ uint8_t s_qm[ACC_Q * ACC_WARPS];
    __shared__ int s_n[ACC_WARPS];
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
    const unsigned below = (1u << lane) - 1u;
    const bool whole = split > 1;   // the block shares an octet
    const int batch = whole ? 32 * ACC_WARPS : 32, self = whole ? (int)threadIdx.x : lane;
    double (*cfq)[25] = s_cf + (whole ? 0 : 32 * wl);
    int *qi = s_qi + (whole ? 0 : ACC_Q * wl);
    uint8_t *qm = s_qm + (whole ? 0 : ACC_Q * wl);
    auto sync = [&]() {
        if (whole) __syncthreads();
        else __syncwarp();
    };
    unsigned long long my_pairs = 0;
    const int per = ACC_WARPS / split;   // octets of a block
    for (int64_t o = (int64_t)blockIdx.x * per + wl / split; o < n_oct; o += (int64_t)gridDim.x * per) {
        const GsProblem &P = BATCH ? probs[mol[o]] : P0;
        Octet q = octet_of(P, level, parents, vmask, o);
        int64_t base[3] = {2 * q.I, 2 * q.J, 2 * q.K};
        double e[3][3];
        float eh[3][3], el[3][3];
        for (int a = 0; a < 3; a++)
            for (int t = 0; t < 3; t++) {
                e[a][t] = gs_lat(P, a, base[a] + t, level);
                double rel = e[a][t] - P.origin[a];
                eh[a][t] = (float)rel;
                el[a][t] = (float)(rel - (double)eh[a][t]);
            }
        double acc[16];
#pragma unroll
        for (int t = 0; t < 16; t++) acc[t] = 0.0;
        int qn = 0, chunk = 0, mine_i = 0;
        unsigned mine_m = 0;   // whole: the candidate tested for the next merge
        const uint8_t vm = q.vmask;
        // update lanes: 4 per (accumulated child, x index); when at most four
        // children are accumulated (a recheck of some cubes of the octet),
        // G groups of lanes take every G-th queued atom and their sums are
        // added at the end, so the FP64 updates issue for several atoms at once
        const int nc = __popc(vm);
        const int gsz = nc <= 1 ? 4 : (nc <= 2 ? 8 : (nc <= 4 ? 16 : 32)), G = 32 / gsz;
        const int pg = lane / gsz, slot = (lane % gsz) >> 2, j = lane & 3;
        int c = -1;
        for (int cc = 0, k = 0; cc < 8; cc++)
            if ((vm >> cc) & 1) {
                if (k == slot) c = gsz == 32 ? (lane >> 2) : cc;
                k++;
            }
        if (gsz == 32) c = lane >> 2;   // every child has its lanes (as without grouping)
        const int cx = c & 1, cy = (c >> 1) & 1, cz = c >> 2;

        // intervals used by the selected children, per axis
        int need[3] = {0, 0, 0};
        for (int cc = 0; cc < 8; cc++)
            if ((vm >> cc) & 1) {
                need[0] |= 1 << (cc & 1);
                need[1] |= 1 << ((cc >> 1) & 1);
                need[2] |= 1 << (cc >> 2);
            }
        auto process = [&](int nproc) {
            if (self < nproc) {
                int i = qi[self];
                double xs[3] = {P.ax[i], P.ay[i], P.az[i]};
                double *cf = cfq[self];
                for (int a = 0; a < 3; a++) coef.axis(xs[a], e[a][0], e[a][1], e[a][2], P.D, cf + 8 * a, need[a]);
                const double w = P.aw[i];
#pragma unroll
                for (int k = 0; k < 8; k++)
                    if ((need[0] >> (k >> 2)) & 1) cf[k] *= w;
            }
            sync();
            if (whole) {
                // the warp's entries: k = wl, in acc[0..3]
                for (int t = pg; t < nproc; t += G) {
                    if (c >= 0 && ((qm[t] >> c) & 1)) {
                        const double *cf = cfq[t];
                        const double wb = cf[4 * cx + j] * cf[8 + 4 * cy + wl];
#pragma unroll
                        for (int l = 0; l < 4; l++) acc[l] = fma(wb, cf[16 + 4 * cz + l], acc[l]);
                    }
                }
            } else {
                for (int t = pg; t < nproc; t += G) {
                    if (c >= 0 && ((qm[t] >> c) & 1)) {
                        const double *cf = cfq[t];
                        double wa = cf[4 * cx + j];
#pragma unroll
                        for (int k = 0; k < 4; k++) {
                            double wb = wa * cf[8 + 4 * cy + k];
#pragma unroll
                            for (int l = 0; l < 4; l++) acc[4 * k + l] = fma(wb, cf[16 + 4 * cz + l], acc[4 * k + l]);
                        }
                    }
                }
            }
            sync();
        };
        // evaluate the queue's first `batch` members once there are so many
        auto drain = [&]() {
            if (qn < batch) return;
            process(batch);
            const int rest = qn - batch;
            int mi = 0;
            uint8_t mm = 0;
            if (self < rest) { mi = qi[batch + self]; mm = qm[batch + self]; }
            sync();
            if (self < rest) { qi[self] = mi; qm[self] = mm; }
            sync();
            qn = rest;
        };
        // whole: queue what the warps found in the last ACC_WARPS chunks, in
        // chunk order (all warps see the same chunks)
        auto merge = [&]() {
            const unsigned bal = __ballot_sync(0xffffffffu, mine_m != 0);
            if (lane == 0) s_n[wl] = __popc(bal);
            __syncthreads();
            int pos = qn + __popc(bal & below);
            for (int v = 0; v < ACC_WARPS; v++) {
                if (v < wl) pos += s_n[v];
                qn += s_n[v];
            }
            if (mine_m) { qi[pos] = mine_i; qm[pos] = (uint8_t)mine_m; }
            mine_m = 0;
            __syncthreads();
            drain();
        };

        // membership of one candidate per lane (i < 0: none): FP32 box
        // distance with a margin, the exact FP64 test (the definition) inside
        // the margin
        auto filter = [&](int i) {
            unsigned m = 0;
            if (i >= 0 && (!whole || chunk % ACC_WARPS == wl)) {
                const float ah[3] = {P.hx[i], P.hy[i], P.hz[i]}, al[3] = {P.lx[i], P.ly[i], P.lz[i]};
                float g2[3][2];
#pragma unroll
                for (int a = 0; a < 3; a++)
#pragma unroll
                    for (int hI = 0; hI < 2; hI++) {
                        float dlo = (eh[a][hI] - ah[a]) + (el[a][hI] - al[a]);
                        float dhi = (ah[a] - eh[a][hI + 1]) + (al[a] - el[a][hI + 1]);
                        float g = fmaxf(0.f, fmaxf(dlo, dhi));
                        g2[a][hI] = g * g;
                    }
                const float R2 = P.fR2[i];
                const float tol = 1e-5f * R2 + 1e-5f;
                unsigned nearm = 0;
#pragma unroll
                for (int cc = 0; cc < 8; cc++) {
                    float d2 = g2[0][cc & 1] + g2[1][(cc >> 1) & 1] + g2[2][cc >> 2];
                    if (d2 < R2 - tol) m |= 1u << cc;
                    else if (d2 <= R2 + tol) nearm |= 1u << cc;
                }
                m &= vm;
                nearm &= vm;
                while (nearm) {
                    const int cc = __ffs(nearm) - 1;
                    nearm &= nearm - 1;
                    double x = P.ax[i], y = P.ay[i], z = P.az[i];
                    double dx = gs_axis_gap(e[0][cc & 1], e[0][(cc & 1) + 1], x);
                    double dy = gs_axis_gap(e[1][(cc >> 1) & 1], e[1][((cc >> 1) & 1) + 1], y);
                    double dz = gs_axis_gap(e[2][cc >> 2], e[2][(cc >> 2) + 1], z);
                    double dd = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
                    if (dd <= P.aR2[i]) m |= 1u << cc;
                }
            }
            my_pairs += __popc(m);
            if (whole) {
                if (m) { mine_i = i; mine_m = m; }
                if (++chunk % ACC_WARPS == 0) merge();
                return;
            }
            unsigned bal = __ballot_sync(0xffffffffu, m != 0);
            int pos = qn + __popc(bal & below);
            if (m) { qi[pos] = i; qm[pos] = (uint8_t)m; }
            qn += __popc(bal);
            __syncwarp();
            drain();
        };

        if (vm) {
            float flo[3] = {eh[0][0], eh[1][0], eh[2][0]}, fhi[3] = {eh[0][2], eh[1][2], eh[2][2]};
            gs_warp_candidates(P, flo, fhi, lane, filter);
            if (chunk % ACC_WARPS != 0) merge();
            if (qn > 0) process(qn);
        }
        for (int off = gsz; off < 32; off <<= 1)
#pragma unroll
            for (int t = 0; t < 16; t++) acc[t] += __shfl_xor_sync(0xffffffffu, acc[t], off);
        if (pg == 0 && c >= 0) {
            double *dst = A_out + ((size_t)o * 8 + c) * 64 + 16 * j;
            if (whole) {
#pragma unroll
                for (int l = 0; l < 4; l++) dst[4 * wl + l] = acc[l];
            } else {
#pragma unroll
                for (int t = 0; t < 16; t++) dst[t] = acc[t];
            }
        }
        if (gsz < 32 && !(whole && wl > 0))   // the children not accumulated hold zeros, as with one lane group
            for (int cc = 0; cc < 8; cc++)
                if (!((vm >> cc) & 1)) {
                    double *z = A_out + ((size_t)o * 8 + cc) * 64;
                    z[lane] = 0.0;
                    z[32 + lane] = 0.0;
                }
    }
    if (pairs) {
        for (int off = 16; off > 0; off >>= 1) my_pairs += __shfl_xor_sync(0xffffffffu, my_pairs, off);
        if (lane == 0 && my_pairs) atomicAdd(pairs, my_pairs);
    }
}

static int grid_for(int64_t n_items, int per_block)
{
    int64_t b = (n_items + per_block - 1) / per_block;
    int64_t cap = 152LL * 64;
    if (b > cap) b = cap;
    return (int)(b < 1 ? 1 : b);
}

int gs_accum_f64(const GsProblem &P, int level, const uint64_t *d_parents, const uint8_t *d_vmask, int64_t n_oct,
                 double *d_A, unsigned long long *d_pairs, cudaStream_t st, cudaEvent_t *ev,
                 const GsProblem *d_probs, const int32_t *d_mol)
{
    if (n_oct <= 0) return GS_OK;
    const double hh = 0.5 * gs_h(P, level);
    if (ev) cudaEventRecord(ev[0], st);
    // up to sixteen octets per SM.  One warp per octet against four (us), the
    // last octets of the finest and of a coarser level of 20,000 atoms cut to
    // length: 152: 124 / 45, 297 / 98; 608: 96 / 88, 233 / 167; 1216: 146 / 152,
    // 396 / 319; 2432: 331 / 284, 752 / 661; 3648: 410 / 423, 1130 / 1026; 7296: 804 /
    // 870, 2190 / 2141; 24,320: 2736 / 3097, 6973 / 7305
    const int split = n_oct <= 152 * 16 ? ACC_WARPS : 1;
    const unsigned grid = grid_for(n_oct, ACC_WARPS / split);
    auto run = [&](auto coef) {
        using C = decltype(coef);
        if (d_probs)
            GS_LAUNCH((k_accum_f64<C, true>), grid, 32 * ACC_WARPS, 0, st)(P, level, d_parents, d_vmask, n_oct, split, coef,
                                                                          d_A, d_pairs, d_probs, d_mol);
        else
            GS_LAUNCH((k_accum_f64<C, false>), grid, 32 * ACC_WARPS, 0, st)(P, level, d_parents, d_vmask, n_oct, split, coef,
                                                                           d_A, d_pairs, nullptr, nullptr);
    };
    // polynomial lengths: a step of one costs 24 of about 330 FP64
    // operations per atom, so the usual needs (7 to 15) have their own
    static const int Ks[] = {7, 8, 9, 10, 12, 15, 20};
    Series S;
    int K = 0;
    if (series_range64(P, hh)) K = series_coeffs(P.D, hh, P.pad, 1e-15, Ks, 7, &S);
#define GS_ACC64(K_)                                                                      \
    case K_: {                                                                            \
        Series64<K_> c;                                                                   \
        c.kappa = S.kappa;                                                                \
        for (int q = 0; q < 4; q++) memcpy(c.c[q], S.c[q], sizeof(double) * K_);          \
        run(c);                                                                           \
        break;                                                                            \
    }
    switch (K) {
        GS_ACC64(7) GS_ACC64(8) GS_ACC64(9) GS_ACC64(10) GS_ACC64(12) GS_ACC64(15) GS_ACC64(20)
    default:
        switch (gq_variant(P.D, hh, false)) {
        case 0: run(Quad64<0, 8>()); break;
        case 1: run(Quad64<1, 16>()); break;
        default: run(Quad64<2, 24>()); break;
        }
    }
#undef GS_ACC64
    if (ev) cudaEventRecord(ev[1], st);
    GS_CHECK(cudaGetLastError());
    return GS_OK;
}

// ---------------------------------------------------------------- estimation
// one cube's 64 coefficients (256 B, 16-byte aligned) in 16-byte loads
__device__ __forceinline__ void load_tensor_f32(const float *__restrict__ src, float *a)
{
    const float4 *s4 = reinterpret_cast<const float4 *>(src);
#pragma unroll
    for (int t = 0; t < 16; t++) {
        const float4 v = __ldg(s4 + t);
        a[4 * t] = v.x; a[4 * t + 1] = v.y; a[4 * t + 2] = v.z; a[4 * t + 3] = v.w;
    }
}

// Truncated SVD bounds of section 2.2.2: FP32 one thread per cube, FP64
// (further down) four lanes or one warp per cube.

template <typename T> __device__ __forceinline__ T t_abs(T x) { return x < T(0) ? -x : x; }
// Jacobi rotation zeroing the inner product ga of two rows with squared
// norms al, be; false when the rows are already orthogonal to within 1e-6
// (the rounding noise of a 16-term dot product is ~1e-6 of |p||q|, so a
// tighter threshold would keep rotating noise until the sweep limit).  The
// rotation only has to reduce ga (the sweep repeats until the threshold
// holds), so the approximate reciprocal, divide and square roots of the SFU
// suffice
__device__ __forceinline__ bool jac_rot(float al, float be, float ga, float &cs, float &sn)
{
    const float e = 1e-6f;
    if (ga == 0.f || ga * ga <= e * e * (al * be)) return false;
    float tau = __fdividef(be - al, 2.f * ga);
    const float at = fabsf(tau);
    float t;
    if (at > 1e18f) {
        t = 0.5f / at;   // 1 / (|tau| + sqrt(1 + tau^2)) without overflowing tau^2
    } else {
        const float q = 1.f + at * at;
        t = __fdividef(1.f, at + q * rsqrtf(q));
    }
    t = copysignf(t, tau);
    cs = rsqrtf(1.f + t * t);
    sn = cs * t;
    return true;
}

// one-sided Jacobi on the 4 rows of X (4 x N): afterwards the rows are
// orthogonal and X_in = Q^T X_out; sv receives their norms (the singular
// values, unsorted)
template <int N>
__device__ __forceinline__ void jacobi_rows(float (&X)[4][N], float (&Q)[4][4], float (&sv)[4])
{
#pragma unroll
    for (int a = 0; a < 4; a++)
#pragma unroll
        for (int b = 0; b < 4; b++) Q[a][b] = a == b ? 1.f : 0.f;
    for (int sweep = 0; sweep < 40; sweep++) {
        bool any = false;
#pragma unroll
        for (int p = 0; p < 3; p++)
#pragma unroll
            for (int q = p + 1; q < 4; q++) {
                float al = 0, be = 0, ga = 0;
                {
                    // FP32: paired (f32x2) products over k = (2m, 2m+1), two
                    // partial sums each to shorten the dependency chains
                    float2 a2[2] = {make_float2(0.f, 0.f), make_float2(0.f, 0.f)};
                    float2 b2[2] = {a2[0], a2[0]}, g2[2] = {a2[0], a2[0]};
#pragma unroll
                    for (int m = 0; m < N / 2; m++) {
                        const float2 xp = make_float2(X[p][2 * m], X[p][2 * m + 1]);
                        const float2 xq = make_float2(X[q][2 * m], X[q][2 * m + 1]);
                        a2[m & 1] = __ffma2_rn(xp, xp, a2[m & 1]);
                        b2[m & 1] = __ffma2_rn(xq, xq, b2[m & 1]);
                        g2[m & 1] = __ffma2_rn(xp, xq, g2[m & 1]);
                    }
                    const float2 a = __fadd2_rn(a2[0], a2[1]), b = __fadd2_rn(b2[0], b2[1]), g = __fadd2_rn(g2[0], g2[1]);
                    al = a.x + a.y;
                    be = b.x + b.y;
                    ga = g.x + g.y;
                }
                float cs, sn;
                if (!jac_rot(al, be, ga, cs, sn)) continue;
                any = true;
                {
                    const float2 c2 = make_float2(cs, cs), s2 = make_float2(sn, sn), ns2 = make_float2(-sn, -sn);
#pragma unroll
                    for (int m = 0; m < N / 2; m++) {
                        const float2 xp = make_float2(X[p][2 * m], X[p][2 * m + 1]);
                        const float2 xq = make_float2(X[q][2 * m], X[q][2 * m + 1]);
                        const float2 np2 = __ffma2_rn(c2, xp, __fmul2_rn(ns2, xq));
                        const float2 nq2 = __ffma2_rn(s2, xp, __fmul2_rn(c2, xq));
                        X[p][2 * m] = np2.x; X[p][2 * m + 1] = np2.y;
                        X[q][2 * m] = nq2.x; X[q][2 * m + 1] = nq2.y;
                    }
#pragma unroll
                    for (int m = 0; m < 2; m++) {
                        const float2 qp = make_float2(Q[p][2 * m], Q[p][2 * m + 1]);
                        const float2 qq = make_float2(Q[q][2 * m], Q[q][2 * m + 1]);
                        const float2 np2 = __ffma2_rn(c2, qp, __fmul2_rn(ns2, qq));
                        const float2 nq2 = __ffma2_rn(s2, qp, __fmul2_rn(c2, qq));
                        Q[p][2 * m] = np2.x; Q[p][2 * m + 1] = np2.y;
                        Q[q][2 * m] = nq2.x; Q[q][2 * m + 1] = nq2.y;
                    }
                }
            }
        if (!any) break;
    }
#pragma unroll
    for (int p = 0; p < 4; p++) {
        float n2 = 0;
#pragma unroll
        for (int k = 0; k < N; k++) n2 += X[p][k] * X[p][k];
        sv[p] = sqrtf(n2);
    }
}

// the SVD of a 4 x 4 matrix: singular values sorted descending in s, the
// matching left vectors in u, the right vectors (normalised rows) in X.  The
// rows are sorted in place by a network of five exchanges.
__device__ __forceinline__ void svd4(float (&X)[4][4], float (&s)[4], float (&u)[4][4])
{
    jacobi_rows<4>(X, u, s);
    auto exchange = [&](int i, int j) {
        const bool sw = s[j] > s[i];
        auto sel = [sw](float &p, float &q) {
            const float a = sw ? q : p, b = sw ? p : q;
            p = a;
            q = b;
        };
        sel(s[i], s[j]);
#pragma unroll
        for (int k = 0; k < 4; k++) {
            sel(X[i][k], X[j][k]);
            sel(u[i][k], u[j][k]);
        }
    };
    exchange(0, 1);
    exchange(2, 3);
    exchange(0, 2);
    exchange(1, 3);
    exchange(1, 2);
#pragma unroll
    for (int p = 0; p < 4; p++) {
        const float inv = s[p] > 0.f ? 1.f / s[p] : 0.f;
#pragma unroll
        for (int k = 0; k < 4; k++) X[p][k] *= inv;
    }
}

// range of sum_j c_j L_j(t) over [-1,1], FP32; the cubic is stationary at the
// derivative's zeros, so approximate divisions serve for these
__device__ __forceinline__ void cubic_range(const float *cf, float &lo, float &hi)
{
    const float p1 = cf[0] + cf[1] + cf[2] + cf[3], m1 = cf[0] - cf[1] + cf[2] - cf[3];
    lo = fminf(p1, m1);
    hi = fmaxf(p1, m1);
    // derivative 3 b3 t^2 + 2 b2 t + b1 in monomials of the cubic
    const float b0 = cf[0] - 0.5f * cf[2], b1 = cf[1] - 1.5f * cf[3], b2 = 1.5f * cf[2], b3 = 2.5f * cf[3];
    const float qa = 3.f * b3, qb = 2.f * b2;
    float r0 = 2.f, r1 = 2.f;   // outside (-1, 1): no zero
    if (qa == 0.f) {
        if (qb != 0.f) r0 = __fdividef(-b1, qb);
    } else {
        const float disc = qb * qb - 4.f * qa * b1;
        if (disc >= 0.f) {
            const float w = -0.5f * (qb + copysignf(sqrtf(disc), qb));
            r0 = w != 0.f ? __fdividef(w, qa) : 0.f;
            if (w != 0.f) r1 = __fdividef(b1, w);
        }
    }
    if (fabsf(r0) < 1.f) {
        const float v = b0 + r0 * (b1 + r0 * (b2 + r0 * b3));
        lo = fminf(lo, v);
        hi = fmaxf(hi, v);
    }
    if (fabsf(r1) < 1.f) {
        const float v = b0 + r1 * (b1 + r1 * (b2 + r1 * b3));
        lo = fminf(lo, v);
        hi = fmaxf(hi, v);
    }
}

template <typename T>
__device__ __forceinline__ int rank99(const T (&s)[4], T &margin)
{
    T tot = s[0] + s[1] + s[2] + s[3];
    T acc = 0;
    T thr = T(0.99) * tot;
    int r = 4;
    margin = tot;
    for (int j = 0; j < 4; j++) {
        acc += s[j];
        T m = t_abs(acc - thr);
        margin = m < margin ? m : margin;
        if (acc >= thr) { r = j + 1; break; }
    }
    return r;
}

// Where the 99% rules could go the other way.  A rule j compares
// sum_{i<=j} s_i with 0.99 sum s; the rules that decide the rank are those up
// to the chosen one, and the one after it (if the chosen rule flipped, the
// next one would decide).  RankNear records the rule nearest its threshold,
// the rank it would give if it flipped, and the second-smallest distance.
struct RankNear {
    float m1, m2;      // smallest and second-smallest distance of a rule from its threshold
    int who;       // -1: outer rule; i >= 0: inner rule of kept term i
    int alt;       // rank that rule gives if it flips (0: none)
    float ssum;        // sum of the outer singular values
};

__device__ __forceinline__ void rank_near(const float (&s)[4], int r, int who, RankNear &rn)
{
    float tot = s[0] + s[1] + s[2] + s[3];
    float acc = 0;
    float thr = 0.99f * tot;
    for (int j = 0; j < 4 && j <= r; j++) {
        acc += s[j];
        float m = t_abs(acc - thr);
        // flipping rule j: below -> rank j+1; at or above -> the next rule decides
        int alt = acc >= thr ? j + 2 : j + 1;
        if (j == 3) alt = 0;
        if (m < rn.m1) {
            rn.m2 = rn.m1;
            rn.m1 = m;
            rn.who = who;
            rn.alt = alt > 4 ? 0 : alt;
        } else if (m < rn.m2) {
            rn.m2 = m;
        }
    }
}

// bounds: out = (L, U, sum|R|, sum|high|, rank, inner ranks); rmargin = the
// smallest distance of a rank rule from its 99% threshold
__device__ __forceinline__ float gap_sens(const float (&s)[4], int kept)
{
    // sum over the kept values of s_i / (distance to the nearest other
    // value): a perturbation E turns the i-th singular pair by about
    // |E| / gap_i, which moves that term's share of the bounds by about
    // s_i |E| / gap_i.  Terms far smaller than their gap contribute little.
    float r = 0.f;
    for (int i = 0; i < kept && i < 4; i++) {
        float g = 1e30f;
        if (i > 0) g = s[i - 1] - s[i];
        if (i < 3) { float d = s[i] - s[i + 1]; g = d < g ? d : g; }
        r += s[i] / (g > 0.f ? g : 1e-30f);
    }
    return r < 1e6f ? r : 1e6f;
}

// fo > 0 forces the outer rank; fi >= 0 forces the inner rank of kept term
// fi to fj; rn (nullable) collects the rules near their thresholds
// A: the tensor (global); S: 80 values of shared memory, EST_THREADS apart
// (the thread's own column), which receive the sorted right and left vectors
// of the outer SVD.  Kept in registers these took 80 of a thread's 243, and
// their rows were picked by selects; 8 warps per SM fitted, now 12 (the
// 1,000,020-atom assembly: 42.6 ms, 32.0 ms).  Four lanes per cube, as in
// FP64, took 53.4 ms: more instructions per cube than the paired FMAs here.
#define EST_THREADS 128
#define EST_SHARED 80
__device__ __forceinline__ void estimate_bounds_sens(const float *A, float *S, float *out, float &rmargin, float &sens, int fo = 0, int fi = -1,
                                                     int fj = 0, RankNear *rn = nullptr);

// element i of four (static indices only, so that arrays stay in registers)
template <typename T>
__device__ __forceinline__ T sel4(int i, T a0, T a1, T a2, T a3)
{
    return i == 0 ? a0 : (i == 1 ? a1 : (i == 2 ? a2 : a3));
}

// The loops over kept terms are rolled, each term's row picked by static selects: one
// copy of the inner SVD and bound code instead of one per possible rank,
// which keeps the kernel within the instruction cache.
__device__ __forceinline__ void estimate_bounds_sens(const float *A, float *S, float *out, float &rmargin, float &sens, int fo, int fi, int fj,
                                                     RankNear *rn)
{
    float s[4];
    float high = 0, tot = 0;
    {
        float X[4][16], Q[4][4], sv[4];
        load_tensor_f32(A, &X[0][0]);
#pragma unroll
        for (int j = 0; j < 4; j++)
#pragma unroll
            for (int k = 0; k < 16; k++) {
                tot += t_abs(X[j][k]);
                if (j >= 2 || (k >> 2) >= 2 || (k & 3) >= 2) high += t_abs(X[j][k]);
            }
        out[3] = high;
        rmargin = 1e30f;
        sens = 0.f;
        if (tot == 0.f) { out[0] = out[1] = out[2] = 0; out[4] = 0; out[5] = 0; return; }
        jacobi_rows<16>(X, Q, sv);
        // row p goes to its place in descending order (equal values in row order)
#pragma unroll
        for (int p = 0; p < 4; p++) {
            int pos = 0;
#pragma unroll
            for (int q = 0; q < 4; q++) pos += (sv[q] > sv[p] || (sv[q] == sv[p] && q < p)) ? 1 : 0;
            const float inv = sv[p] > 0.f ? 1.f / sv[p] : 0.f;
            float *row = S + 16 * pos * EST_THREADS, *left = S + (64 + 4 * pos) * EST_THREADS;
#pragma unroll
            for (int k = 0; k < 16; k++) row[k * EST_THREADS] = X[p][k] * inv;
#pragma unroll
            for (int k = 0; k < 4; k++) left[k * EST_THREADS] = Q[p][k];
#pragma unroll
            for (int i = 0; i < 4; i++)
                if (pos == i) s[i] = sv[p];
        }
    }
    float rm;
    int jr = rank99(s, rm);
    if (fo > 0) {
        jr = fo;
        rm = 1e30f;
    } else if (rn) {
        rn->ssum = s[0] + s[1] + s[2] + s[3];
        rank_near(s, jr, -1, *rn);
    }
    rmargin = rm;
    sens = gap_sens(s, jr);
    // R = A minus the kept rank-one terms, subtracted in place
    float R[64];
    load_tensor_f32(A, R);
    float M = 0, m = 0;
    int inner = 0;
#pragma unroll 1
    for (int i = 0; i < jr; i++) {
        float V[4][4], d[4], w[4][4], ui[4];
        const float *row = S + 16 * i * EST_THREADS, *left = S + (64 + 4 * i) * EST_THREADS;
#pragma unroll
        for (int k = 0; k < 4; k++)
#pragma unroll
            for (int l = 0; l < 4; l++) V[k][l] = row[(4 * k + l) * EST_THREADS];
#pragma unroll
        for (int a = 0; a < 4; a++) ui[a] = left[a * EST_THREADS];
        const float si0 = sel4(i, s[0], s[1], s[2], s[3]);
        svd4(V, d, w);
        float rmi;
        int ji = rank99(d, rmi);
        if (i == fi) {
            ji = fj;
        } else {
            rmargin = rmi < rmargin ? rmi : rmargin;
            if (rn) rank_near(d, ji, i, *rn);
        }
        float si = gap_sens(d, ji);
        sens = si > sens ? si : sens;
        inner += ji;
        float Myz = 0, myz = 0;
#pragma unroll 1
        for (int k = 0; k < ji; k++) {
            float wk[4], Vk[4];
#pragma unroll
            for (int b = 0; b < 4; b++) {
                wk[b] = sel4(k, w[0][b], w[1][b], w[2][b], w[3][b]);
                Vk[b] = sel4(k, V[0][b], V[1][b], V[2][b], V[3][b]);
            }
            const float dk = sel4(k, d[0], d[1], d[2], d[3]);
            float ly, hy, lz, hz;
            cubic_range(wk, ly, hy);
            cubic_range(Vk, lz, hz);
            float p0 = hy * hz, p1 = hy * lz, p2 = ly * hz, p3 = ly * lz;
            float pmx = p0, pmn = p0;
            pmx = p1 > pmx ? p1 : pmx; pmn = p1 < pmn ? p1 : pmn;
            pmx = p2 > pmx ? p2 : pmx; pmn = p2 < pmn ? p2 : pmn;
            pmx = p3 > pmx ? p3 : pmx; pmn = p3 < pmn ? p3 : pmn;
            Myz += dk * pmx;
            myz += dk * pmn;
            float sd = si0 * dk;
#pragma unroll
            for (int a = 0; a < 4; a++) {
                float sa = sd * ui[a];
#pragma unroll
                for (int b = 0; b < 4; b++) {
                    float sab = sa * wk[b];
#pragma unroll
                    for (int cc = 0; cc < 4; cc++) R[16 * a + 4 * b + cc] -= sab * Vk[cc];
                }
            }
        }
        float lx, hx;
        cubic_range(ui, lx, hx);
        float p0 = hx * Myz, p1 = hx * myz, p2 = lx * Myz, p3 = lx * myz;
        float pmx = p0, pmn = p0;
        pmx = p1 > pmx ? p1 : pmx; pmn = p1 < pmn ? p1 : pmn;
        pmx = p2 > pmx ? p2 : pmx; pmn = p2 < pmn ? p2 : pmn;
        pmx = p3 > pmx ? p3 : pmx; pmn = p3 < pmn ? p3 : pmn;
        M += si0 * pmx;
        m += si0 * pmn;
    }
    float sr = 0;
#pragma unroll
    for (int t = 0; t < 64; t++) sr += t_abs(R[t]);
    out[0] = m - sr;
    out[1] = M + sr;
    out[2] = sr;
    out[4] = (float)jr;
    out[5] = (float)inner;
}

template <typename T>
__device__ __forceinline__ int decide(const T *b, T c, T precision, int level, int max_depth)
{
    if (b[4] == T(0)) return DEC_DISCARD;
    if (!(b[0] <= c && c <= b[1])) return DEC_DISCARD;
    if (b[3] <= precision) return DEC_ACCEPT;
    if (level >= max_depth) return DEC_FORCED;
    return DEC_SPLIT;
}

// P~ at the 8 cube corners: L_n(+-1) = (+-1)^n, so each corner value is a
// signed sum of the coefficients; lo and hi receive the smallest and largest
template <typename T>
__device__ __forceinline__ void corner_range(const T *a, T &lo, T &hi)
{
    lo = T(3.0e38);
    hi = T(-3.0e38);
#pragma unroll
    for (int sx = 0; sx < 2; sx++) {
        T bx[16];
#pragma unroll
        for (int kl = 0; kl < 16; kl++) {
            const T e = a[kl] + a[32 + kl], o = a[16 + kl] + a[48 + kl];
            bx[kl] = sx ? e + o : e - o;
        }
#pragma unroll
        for (int sy = 0; sy < 2; sy++) {
            T cz[4];
#pragma unroll
            for (int l = 0; l < 4; l++) {
                const T e = bx[l] + bx[8 + l], o = bx[4 + l] + bx[12 + l];
                cz[l] = sy ? e + o : e - o;
            }
            const T e = cz[0] + cz[2], o = cz[1] + cz[3];
            lo = fmin(lo, fmin(e - o, e + o));
            hi = fmax(hi, fmax(e - o, e + o));
        }
    }
}

// Range of P~ over the cube from its trilinear part's corner values and the
// sum `high` of the other coefficients' sizes, and the distance e of the
// tensor from a rank-one tensor (the one through its three fibres at 000):
// what proves a discard without the SVD.  For any tensor within e of rank one,
//   U <= max P~ + 53 e,   L >= min P~ - 53 e
// hold for the bounds of the two-level truncated SVD, whatever its ranks: let
// T = s_1 d_11 u_1 w_11 v_11 be its leading term and S the sum of the other
// terms' s_i d_ik.  |u|, |w|, |v| <= 2 on the interval (unit vectors of four
// Legendre coefficients), so every other term adds at most 8 s_i d_ik to U,
// kept (through its range) or dropped (through sum|R|): U <= max T + 8 S.
// sum_k d_1k over k >= 2 is at most sqrt(3) times their norm, which is at most
// e / s_1 (the distance of u_1^T A from rank one); sum_i s_i over i >= 2 at most
// sqrt(3) e (the distance of the unfolding from rank one) and sum_k d_ik <= 2:
// S <= 3 sqrt(3) e.  And max T <= max P~ + sum|A - T| <= max P~ + 8 |A - T|,
// |A - T| <= sqrt(2) e.  8 sqrt(2) + 24 sqrt(3) = 52.9.
// On the levels of a molecule 25 to 75% of the cubes that neither straddle c
// nor lack atoms are discarded so: the SVD pass of 1,000,020 atoms in FP32 32.0 ->
// 26.2 ms at 1.9 ms more in the first pass, of 20,000 atoms in FP64 19.1 -> 16.2
// at 1.3 more.
template <typename T>
__device__ __forceinline__ void trilinear_range(const T *a, T high, T &mn, T &mx)
{
    // coefficients (j, k, l) in {0, 1}: |L_1| = 1 at the corners
    T lo = T(3.0e38), hi = T(-3.0e38);
#pragma unroll
    for (int c = 0; c < 4; c++) {
        const T y = (c & 1) ? T(1) : T(-1), z = (c & 2) ? T(1) : T(-1);
        const T e = (a[0] + y * a[4]) + z * (a[1] + y * a[5]);
        const T o = fabs((a[16] + y * a[20]) + z * (a[17] + y * a[21]));
        lo = fmin(lo, e - o);
        hi = fmax(hi, e + o);
    }
    mn = lo - high;
    mx = hi + high;
}
// squared distance from the rank-one tensor; a[0] != 0.  Its squares lose
// their precision below 1e-38 (FP32) and 1e-308 (FP64), so it is compared only
// with the square of a room above 1e-17 or 1e-150 (at an isovalue of 1e-20 the
// FP32 form otherwise drops cubes that the SVD keeps)
template <typename T>
__device__ __forceinline__ T rank_one_dist2(const T *a)
{
    const T inv = T(1) / a[0];
    T d2 = T(0), ez[4];
#pragma unroll
    for (int l = 0; l < 4; l++) ez[l] = a[l] * inv;
#pragma unroll
    for (int j = 0; j < 4; j++)
#pragma unroll
        for (int k = 0; k < 4; k++) {
            const T xy = a[16 * j] * (a[4 * k] * inv);
#pragma unroll
            for (int l = 0; l < 4; l++) {
                const T t = a[16 * j + 4 * k + l] - xy * ez[l];
                d2 += t * t;
            }
        }
    return d2;
}
#define RANK_ONE_SLOPE 53

// Literal order of steps 2 and 3: a child whose higher-order coefficients
// meet the bound is accepted before its bounds are tested; a root cube that
// passes the bound test is divided.
__device__ __forceinline__ int decide_literal(const double *b, double c, double precision, int level, int max_depth)
{
    if (b[4] == 0.0) return DEC_DISCARD;
    if (level > 0 && b[3] <= precision) return DEC_ACCEPT;
    if (!(b[0] <= c && c <= b[1])) return DEC_DISCARD;
    if (level >= max_depth) return DEC_FORCED;
    return DEC_SPLIT;
}

// size of the higher-than-linear coefficients: largest magnitude (GS_NORM_MAX)
// or root sum of squares (GS_NORM_RSS); the sum of magnitudes is b[3] already
__device__ __forceinline__ double high_norm(const double *a, int norm)
{
    double mx = 0.0, ss = 0.0;
    for (int j = 0; j < 4; j++)
        for (int k = 0; k < 4; k++)
            for (int l = 0; l < 4; l++)
                if (j >= 2 || k >= 2 || l >= 2) {
                    const double v = a[16 * j + 4 * k + l];
                    mx = fmax(mx, fabs(v));
                    ss = fma(v, v, ss);
                }
    return norm == GS_NORM_MAX ? mx : sqrt(ss);
}

// ---- the FP64 estimate: four lanes per cube
// GB300 issues one FP64 warp instruction per SM every 16 cycles, so the FP64
// estimate is bound by their number, and by their latency when few cubes are
// listed.  Lane l of a quad holds the entries (x, y, z) = (j, k, l) of its
// cube: its 4 columns of the 4 x 16 unfolding, and afterwards column l of
// each right vector V_i, so the inner SVDs need no data moved.  The state
// stays in registers (one thread per cube spilled 3.7 KB) and only 8 cubes
// share a warp's loops.  A 20,000-atom FP64 mesh: 23.3 ms with one thread per
// cube and FP64 divisions and roots in every rotation, 19.1 ms.

// gross FP64 approximations (about 20 bits) of the special-function unit
__device__ __forceinline__ double rcp64_approx(double x)
{
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    return y;
}
__device__ __forceinline__ double rsqrt64_approx(double x)
{
    double y;
    asm("rsqrt.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(x));
    return y;
}
// 1/x to about 40 bits
__device__ __forceinline__ double rcp64_40(double x)
{
    const double y = rcp64_approx(x);
    return fma(y, fma(-x, y, 1.0), y);
}
// 1/sqrt(x) to FP64 rounding: the approximation y0 (relative error below
// 2^-18) times the series of (1 - e)^(-1/2), e = 1 - x y0^2, to e^3 (the
// rest is below 2^-70)
__device__ __forceinline__ double rsqrt64(double x)
{
    const double y0 = rsqrt64_approx(x);
    const double e = fma(-x, y0 * y0, 1.0);
    return fma(y0 * e, fma(e, fma(e, 0.3125, 0.375), 0.5), y0);
}

// The rotation that makes rows with squared norms al, be and inner product
// ga orthogonal, as tan(a/2) and sin(a) of three shears (p -= th q,
// q += sn p, p -= th q), and the norms after it.  With h = ga / (be - al),
// tan(a) = 2 h / (1 + sqrt(1 + 4 h^2)).  The angle only has to reduce ga (the
// sweep repeats until the threshold holds): small ones, which the later
// sweeps consist of, are taken to 40 bits, so that convergence stays
// quadratic, large ones in FP32.  The shears are orthonormal to FP64 for any
// th as long as sn = 2 th / (1 + th^2) holds to FP64: the series in th^2
// (th^6 < 2e-22), or the reciprocal approximation and its series to e^2 (the
// rest is below 2^-54).
__device__ __forceinline__ void jac_shears64(double &al, double &be, double ga, double &th, double &sn)
{
    const double df = be - al, rc = rcp64_approx(df);
    double h = ga * rc;
    if (__double2hiint(fabs(h)) < 0x3f400000) {   // |h| < 2^-11
        h = fma(h, fma(-df, rc, 1.0), h);
        const double h2 = h * h;
        th = h * fma(-0.625, h2, 0.5);
        const double t2 = th * th, tt = th + th;
        sn = fma(tt, fma(t2, t2, -t2), tt);
    } else {
        const float hf = copysignf(fminf(fabsf((float)h), 1e9f), (float)h), q = fmaf(4.f * hf, hf, 1.f);
        const float tf = __fdividef(2.f * hf, fmaf(q, rsqrtf(q), 1.f));
        const float r = fmaf(tf, tf, 1.f);
        h = (double)tf;
        th = (double)__fdividef(tf, fmaf(r, rsqrtf(r), 1.f));
        const double rr = fma(th, th, 1.0), y0 = rcp64_approx(rr), e = fma(-rr, y0, 1.0);
        sn = (th + th) * fma(y0, fma(e, e, e), y0);
    }
    al = fma(-h, ga, al);
    be = fma(h, ga, be);
}
// |ga| > 1e-15 sqrt(al be), on the exponents and leading mantissa bits as a
// piecewise linear logarithm (within 13% on the threshold), which keeps the
// test off the FP64 pipe
__device__ __forceinline__ bool jac_needed64(double al, double be, double ga)
{
    const int bias = 0x3ff00000;
    const int lg = (__double2hiint(ga) & 0x7fffffff) - bias;
    const int la = max(__double2hiint(al), 0) - bias, lb = max(__double2hiint(be), 0) - bias;
    return lg > -(900 << 20) && 2ll * lg > (long long)la + lb - 104500000ll;   // 2 log2(1e-15) 2^20
}

// The two kernels of the FP64 estimate take every sum in the same order and
// round it alike, so a cube's bounds do not depend on which of them (the
// length of the list) it meets.  A sum over the 16 columns (k, l) of the
// unfolding adds fused products over k, then pairs over l; one over all 64
// entries adds pairs over the rows 2h, 2h + 1, over k, over h and over l.
// Products and additions that a compiler could contract either way are
// written as rounded ones.

// the sum over the quad of its lanes' parts
__device__ __forceinline__ double quad_sum(double v)
{
    const unsigned full = 0xffffffffu;
    v = __dadd_rn(v, __shfl_xor_sync(full, v, 1));
    return __dadd_rn(v, __shfl_xor_sync(full, v, 2));
}
// the lane's part of the inner product of two rows
template <int NC>
__device__ __forceinline__ double row_dot(const double (&a)[NC], const double (&b)[NC])
{
    double v = __dmul_rn(a[0], b[0]);
#pragma unroll
    for (int k = 1; k < NC; k++) v = fma(a[k], b[k], v);
    return v;
}
// the lane's part of a sum over all entries v[j][k]
__device__ __forceinline__ double entry_sum(const double (&v)[4][4])
{
    double t[2];
#pragma unroll
    for (int h = 0; h < 2; h++)
        t[h] = __dadd_rn(__dadd_rn(__dadd_rn(v[2 * h][0], v[2 * h + 1][0]), __dadd_rn(v[2 * h][1], v[2 * h + 1][1])),
                         __dadd_rn(__dadd_rn(v[2 * h][2], v[2 * h + 1][2]), __dadd_rn(v[2 * h][3], v[2 * h + 1][3])));
    return __dadd_rn(t[0], t[1]);
}

// Squares of the entries and their products leave FP64's range for isovalues
// below about 1e-130: a tensor whose sum of magnitudes lies outside 2^-300 ..
// 2^300 is scaled by a power of two (exactly), and its bounds scaled back.
// False: no scaling, and both factors are 1.
__device__ __forceinline__ bool svd_scale64(double tot, double &to, double &back)
{
    const int e = (__double2hiint(tot) >> 20) & 0x7ff;
    const bool out = (e < 723 || e > 1323) && tot != 0.0 && e < 2046;
    to = out ? __hiloint2double((2046 - (e ? e : 1)) << 20, 0) : 1.0;
    back = out ? __hiloint2double((e ? e : 1) << 20, 0) : 1.0;
    return out;
}

// one-sided Jacobi on the 4 rows of a matrix whose columns lie in the four
// lanes of a quad (NC each): y the lane's columns, z its column of the
// accumulated rotations (initially the identity).  Each of the three rounds
// of a sweep rotates two disjoint row pairs; the lane's lowest bit selects
// the pair whose angle it finds.  Squared norms are taken anew at every sweep
// and follow the rotations within it (they only steer).  All 32 lanes take
// part; act: this quad still has work to do.
template <int NC>
__device__ __forceinline__ void jacobi_quad(double (&y)[4][NC], double (&z)[4], bool act, int lane)
{
    const unsigned full = 0xffffffffu;
    const bool odd = lane & 1;
#pragma unroll 1
    for (int sweep = 0; sweep < 40; sweep++) {
        double n[4];
#pragma unroll
        for (int p = 0; p < 4; p++) n[p] = quad_sum(row_dot(y[p], y[p]));
        bool any = false;
#pragma unroll
        for (int round = 0; round < 3; round++) {
            // (0,1)(2,3), (0,2)(1,3), (0,3)(1,2)
            const int q0 = round + 1, p1 = round == 0 ? 2 : 1, q1 = round == 2 ? 2 : 3;
            const double g0 = row_dot(y[0], y[q0]), g1 = row_dot(y[p1], y[q1]);
            // the lane's pair: sum over the quad of its inner product
            double ga = __dadd_rn(odd ? g1 : g0, __shfl_xor_sync(full, odd ? g0 : g1, 1));
            ga = __dadd_rn(ga, __shfl_xor_sync(full, ga, 2));
            double al = odd ? n[p1] : n[0], be = odd ? n[q1] : n[q0];
            const bool rot = act && jac_needed64(al, be, ga);
            if (!__any_sync(full, rot)) continue;
            any |= rot;
            double th = 0.0, sn = 0.0;
            if (rot) jac_shears64(al, be, ga, th, sn);
            // both pairs' rotations and norms
            const double tho = __shfl_xor_sync(full, th, 1), sno = __shfl_xor_sync(full, sn, 1);
            const double alo = __shfl_xor_sync(full, al, 1), beo = __shfl_xor_sync(full, be, 1);
            const double t0 = odd ? tho : th, s0 = odd ? sno : sn, t1 = odd ? th : tho, s1 = odd ? sn : sno;
            n[0] = odd ? alo : al;
            n[q0] = odd ? beo : be;
            n[p1] = odd ? al : alo;
            n[q1] = odd ? be : beo;
            auto turn = [](double &p, double &q, double t, double s) {
                p = fma(-t, q, p);
                q = fma(s, p, q);
                p = fma(-t, q, p);
            };
#pragma unroll
            for (int k = 0; k < NC; k++) {
                turn(y[0][k], y[q0][k], t0, s0);
                turn(y[p1][k], y[q1][k], t1, s1);
            }
            turn(z[0], z[q0], t0, s0);
            turn(z[p1], z[q1], t1, s1);
        }
        if (!__any_sync(full, any)) break;
    }
}

// singular values (norms of the rows), rows sorted by descending value (equal
// ones in row order) and normalised, the accumulated rotations alike
template <int NC>
__device__ __forceinline__ void svd_order_quad(double (&y)[4][NC], double (&z)[4], double (&s)[4], int lane)
{
    const unsigned full = 0xffffffffu;
    double n[4], sv[4], inv[4];
#pragma unroll
    for (int p = 0; p < 4; p++) n[p] = quad_sum(row_dot(y[p], y[p]));
    // one root per lane, passed around the quad
    const double nm = sel4(lane & 3, n[0], n[1], n[2], n[3]);
    const double im = nm > 1e-290 ? rsqrt64(nm) : 0.0, sm = nm * im;
#pragma unroll
    for (int p = 0; p < 4; p++) {
        sv[p] = __shfl_sync(full, sm, p, 4);
        inv[p] = __shfl_sync(full, im, p, 4);
    }
    double ys[4][NC], zs[4];
    int pos[4];
#pragma unroll
    for (int p = 0; p < 4; p++) {
        pos[p] = 0;
#pragma unroll
        for (int q = 0; q < 4; q++) {
            // (non-negative: ordered as their bits)
            const long long a = __double_as_longlong(sv[q]), b = __double_as_longlong(sv[p]);
            pos[p] += (a > b || (a == b && q < p)) ? 1 : 0;
        }
#pragma unroll
        for (int k = 0; k < NC; k++) y[p][k] *= inv[p];
    }
#pragma unroll
    for (int i = 0; i < 4; i++)
#pragma unroll
        for (int p = 0; p < 4; p++)
            if (pos[p] == i) {
                s[i] = sv[p];
                zs[i] = z[p];
#pragma unroll
                for (int k = 0; k < NC; k++) ys[i][k] = y[p][k];
            }
#pragma unroll
    for (int i = 0; i < 4; i++) {
        z[i] = zs[i];
#pragma unroll
        for (int k = 0; k < NC; k++) y[i][k] = ys[i][k];
    }
}

// rows <-> lanes of a 4 x 4 matrix held one column per lane of a quad
__device__ __forceinline__ void transpose_quad(const double (&v)[4], double (&o)[4], int lane)
{
    const unsigned full = 0xffffffffu;
    const bool b0 = lane & 1, b1 = lane & 2;
    // swap the off-diagonal elements of the 2 x 2 blocks, then the blocks
    const double x0 = __shfl_xor_sync(full, b0 ? v[0] : v[1], 1), x1 = __shfl_xor_sync(full, b0 ? v[2] : v[3], 1);
    const double a0 = b0 ? x0 : v[0], a1 = b0 ? v[1] : x0, a2 = b0 ? x1 : v[2], a3 = b0 ? v[3] : x1;
    const double y0 = __shfl_xor_sync(full, b1 ? a0 : a2, 2), y1 = __shfl_xor_sync(full, b1 ? a1 : a3, 2);
    o[0] = b1 ? y0 : a0;
    o[1] = b1 ? y1 : a1;
    o[2] = b1 ? a2 : y0;
    o[3] = b1 ? a3 : y1;
}

// range of sum_j c_j L_j(t) over [-1,1] as cubic_range<T> gives it; the
// derivative's zeros are taken to about 40 bits, which the cubic's values
// there, being stationary, do not feel
__device__ __forceinline__ void cubic_range64(const double (&cf)[4], double &lo, double &hi)
{
    const double e = cf[0] + cf[2], o = cf[1] + cf[3];
    lo = e - fabs(o);
    hi = e + fabs(o);
    const double b0 = fma(-0.5, cf[2], cf[0]), b1 = fma(-1.5, cf[3], cf[1]), b3 = 2.5 * cf[3];
    const double b2 = fma(1.5, cf[2], 0.0);   // (a zero without its sign, which a rotation by nothing may turn)
    // derivative / 1: 3 b3 t^2 + 2 b2 t + b1; half discriminant b2^2 - 3 b3 b1
    const double qa = 3.0 * b3;
    const double disc = fma(b2, b2, -qa * b1);
    double r0 = 2.0, r1 = 2.0;   // outside [-1, 1]: no root
    if (qa == 0.0) {
        if (b2 != 0.0) r0 = -0.5 * b1 * rcp64_40(b2);
    } else if (disc >= 0.0) {
        double sq = 0.0;
        if (disc > 1e-290) {
            const double g = rsqrt64_approx(disc);
            sq = disc * g;
            sq = fma(0.5 * g, fma(-sq, sq, disc), sq);
        }
        const double w = -(b2 + copysign(sq, b2));
        if (w != 0.0) {
            r0 = w * rcp64_40(qa);
            r1 = b1 * rcp64_40(w);
        } else {
            r0 = 0.0;
        }
    }
    if ((__double2hiint(r0) & 0x7fffffff) < 0x3ff00000) {   // |r0| < 1
        const double v = fma(r0, fma(r0, fma(r0, b3, b2), b1), b0);
        lo = fmin(lo, v);
        hi = fmax(hi, v);
    }
    if ((__double2hiint(r1) & 0x7fffffff) < 0x3ff00000) {
        const double v = fma(r1, fma(r1, fma(r1, b3, b2), b1), b0);
        lo = fmin(lo, v);
        hi = fmax(hi, v);
    }
}

// range of a product of two independent factors
__device__ __forceinline__ void product_range(double l1, double h1, double l2, double h2, double &mn, double &mx)
{
    const double p0 = h1 * h2, p1 = h1 * l2, p2 = l1 * h2, p3 = l1 * l2;
    mx = fmax(fmax(p0, p1), fmax(p2, p3));
    mn = fmin(fmin(p0, p1), fmin(p2, p3));
}

#define E64W_WARPS 4
// The most cubes k_estimate_f64w takes.  Its time grows by a step every 608
// cubes (four warps per SM), that of k_estimate_f64 not before 4864.  The two
// in us on lists of the finest and the coarsest level of 20,000 atoms cut to
// length: 608: 47 / 88, 55 / 162; 1216: 69 / 90, 80 / 161; 1536: 98 / 92, 113 / 162; 2128:
// 126 / 91, 149 / 162; 3040: 157 / 90, 186 / 163
#define E64W_MAX 1536

// the decision of cube q from its bounds, and the counts of small margins
__device__ __forceinline__ void finish_f64(const GsProblem &P, int level, int64_t q, const double *a,
                                           const double (&b0)[6], double rrel, uint8_t *dec, double *bounds)
{
    double b[6];
#pragma unroll
    for (int k = 0; k < 6; k++) b[k] = b0[k];
    if (P.norm != GS_NORM_SUM) b[3] = high_norm(a, P.norm);
    const int d = P.order == GS_ORDER_LITERAL ? decide_literal(b, P.c, P.precision, level, P.max_depth)
                                              : decide<double>(b, P.c, P.precision, level, P.max_depth);
    dec[q] = (uint8_t)d;
    if (P.near && b[4] != 0.0) {
        // the margins of the decision against its thresholds
        const double scale = fabs(P.c) + fabs(b[0]) + fabs(b[1]);
        if (fmin(fabs(P.c - b[0]), fabs(b[1] - P.c)) < GS_NEAR_REL * scale) atomicAdd(&P.near[0], 1ull);
        if (d != DEC_DISCARD && fabs(P.precision - b[3]) < GS_NEAR_REL * (P.precision + b[3]))
            atomicAdd(&P.near[1], 1ull);
        if (rrel < GS_NEAR_REL) atomicAdd(&P.near[2], 1ull);
    }
    if (bounds)
        for (int k = 0; k < 6; k++) bounds[q * 6 + k] = b[k];
}

__global__ void __launch_bounds__(128) k_estimate_f64(GsProblem P, int level, const double *__restrict__ A,
                                                      int64_t n, const uint64_t *parents, const uint8_t *vmask,
                                                      uint8_t *__restrict__ dec, double *__restrict__ bounds,
                                                      const int32_t *__restrict__ list, const unsigned *nlist)
{
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, l = lane & 3;
    // a compacted list of the cubes to estimate, or all of them
    const int64_t cnt = list ? (int64_t)*nlist : n;
    if (cnt <= E64W_MAX) return;   // k_estimate_f64w takes them
    const int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 2;
    if (t - (lane >> 2) >= cnt) return;   // the whole warp is past the end
    int64_t q = -1;
    if (t < cnt) {
        q = list ? (int64_t)list[t] : t;
        const Octet oc = octet_of(P, level, parents, vmask, q >> 3);
        if (!((oc.vmask >> (q & 7)) & 1)) {
            if (l == 0) dec[q] = DEC_INVALID;
            q = -1;
        }
    }
    const double *a = A + (q >= 0 ? q * 64 : 0) + l;
    double y[4][4], z[4], tot, high;
    {
        double v[4][4];
#pragma unroll
        for (int j = 0; j < 4; j++) {
            z[j] = j == l ? 1.0 : 0.0;
#pragma unroll
            for (int k = 0; k < 4; k++) {
                y[j][k] = q >= 0 ? a[16 * j + 4 * k] : 0.0;
                v[j][k] = fabs(y[j][k]);
            }
        }
        tot = quad_sum(entry_sum(v));
#pragma unroll
        for (int j = 0; j < 2; j++)
#pragma unroll
            for (int k = 0; k < 2; k++)
                if (l < 2) v[j][k] = 0.0;
        high = quad_sum(entry_sum(v));
    }
    double to, back;
    const bool scaled = __any_sync(full, svd_scale64(tot, to, back));
    if (scaled)
#pragma unroll
        for (int j = 0; j < 4; j++)
#pragma unroll
            for (int k = 0; k < 4; k++) y[j][k] *= to;
    double s[4], rm = 0.0, rrel = 1e30;
    jacobi_quad<4>(y, z, true, lane);
    svd_order_quad<4>(y, z, s, lane);
    int jr = 0;
    if (tot != 0.0) {
        jr = rank99(s, rm);
        rrel = rm / (s[0] + s[1] + s[2] + s[3]);
    }
    // the residual A minus the kept rank-one terms, same layout as y
    double R[4][4];
#pragma unroll
    for (int j = 0; j < 4; j++)
#pragma unroll
        for (int k = 0; k < 4; k++) R[j][k] = q >= 0 ? a[16 * j + 4 * k] : 0.0;
    if (scaled)
#pragma unroll
        for (int j = 0; j < 4; j++)
#pragma unroll
            for (int k = 0; k < 4; k++) R[j][k] *= to;
    double lx, hx;   // lane l: the range of u_l
    {
        double cf[4];
        transpose_quad(z, cf, lane);   // lane l: u_l[0..3] (z[i] of lane b is u_i[b])
        cubic_range64(cf, lx, hx);
    }
    double M = 0.0, m = 0.0;
    int inner = 0;
    const int jmax = __reduce_max_sync(full, jr);
#pragma unroll 1
    for (int i = 0; i < jmax; i++) {
        const bool on = i < jr;
        double v[4][1], w[4], d[4];
#pragma unroll
        for (int k = 0; k < 4; k++) {
            v[k][0] = on ? sel4(i, y[0][k], y[1][k], y[2][k], y[3][k]) : 0.0;
            w[k] = k == l ? 1.0 : 0.0;
        }
        jacobi_quad<1>(v, w, on, lane);
        svd_order_quad<1>(v, w, d, lane);
        const double si = sel4(i, s[0], s[1], s[2], s[3]);
        int ji = 0;
        if (on) {
            double rmi;
            ji = rank99(d, rmi);
            rrel = fmin(rrel, rmi / (d[0] + d[1] + d[2] + d[3]));
        }
        inner += ji;
        // lane k: the ranges of w_k and V_k
        double cf[4], vr[4], lo, hi, lo2, hi2, mn, mx;
        transpose_quad(w, cf, lane);
        cubic_range64(cf, lo, hi);
#pragma unroll
        for (int k = 0; k < 4; k++) vr[k] = v[k][0];
        transpose_quad(vr, cf, lane);
        cubic_range64(cf, lo2, hi2);
        product_range(lo, hi, lo2, hi2, mn, mx);
        const double dl = sel4(l, d[0], d[1], d[2], d[3]);
        const double Myz = quad_sum(l < ji ? __dmul_rn(dl, mx) : 0.0);
        const double myz = quad_sum(l < ji ? __dmul_rn(dl, mn) : 0.0);
        product_range(__shfl_sync(full, lx, i, 4), __shfl_sync(full, hx, i, 4), myz, Myz, mn, mx);
        if (on) {
            M = fma(si, mx, M);
            m = fma(si, mn, m);
        }
        const double zi = sel4(i, z[0], z[1], z[2], z[3]);
        double u[4];
#pragma unroll
        for (int j = 0; j < 4; j++) u[j] = __shfl_sync(full, zi, j, 4);
        const int kmax = __reduce_max_sync(full, ji);
#pragma unroll 1
        for (int k = 0; k < kmax; k++) {
            const double wk = sel4(k, w[0], w[1], w[2], w[3]), vk = sel4(k, vr[0], vr[1], vr[2], vr[3]);
            const double dk = sel4(k, d[0], d[1], d[2], d[3]);
            const double x = k < ji ? si * dk * vk : 0.0;
#pragma unroll
            for (int b = 0; b < 4; b++) {
                const double xw = x * __shfl_sync(full, wk, b, 4);
#pragma unroll
                for (int j = 0; j < 4; j++) R[j][b] = fma(-u[j], xw, R[j][b]);
            }
        }
    }
#pragma unroll
    for (int j = 0; j < 4; j++)
#pragma unroll
        for (int k = 0; k < 4; k++) R[j][k] = fabs(R[j][k]);
    const double sr = quad_sum(entry_sum(R));
    if (q < 0 || l != 0) return;
    const double b[6] = {(m - sr) * back, (M + sr) * back, sr * back, high, (double)jr, (double)inner};
    finish_f64(P, level, q, a, b, rrel, dec, bounds);
}

// ---- few cubes: one warp per cube
// A warp of the kernel above spends some 1500 FP64 instructions, each 64
// cycles of its SM quarter, however few of its quads hold a cube.  With a
// cube per warp that is about half: 16 lanes hold one column of the
// unfolding each, half the warp one row pair of the round and its angle (the
// rows change places between the halves), and the inner SVDs of the four
// right vectors run side by side, 8 lanes each.  The recheck of a 523-atom
// mixed mesh (4 levels of up to 100 cubes): 2130 us with one thread per cube,
// 503 us with quads, 184 us.

// the inner product of two rows with one column per lane, 4 (LC = 2) or 16
// (LC = 4, column 4 k + l) of them, in the order of row_dot and quad_sum
template <int LC>
__device__ __forceinline__ double row_dot_warp(double p, double q, int lane)
{
    const unsigned full = 0xffffffffu;
    double v = __dmul_rn(p, q);
    if (LC == 4) {
        const int k = (lane >> 2) & 3;
#pragma unroll
        for (int s = 1; s < 4; s++) {
            const double t = fma(p, q, __shfl_up_sync(full, v, 4));
            if (k == s) v = t;
        }
        v = __shfl_sync(full, v, lane | 12);
    }
    return quad_sum(v);
}
// the sum over the warp of all entries, lane (h, k, l) holding the sum of
// those of the rows 2h and 2h + 1, in the order of entry_sum and quad_sum
__device__ __forceinline__ double entry_sum_warp(double v)
{
    const unsigned full = 0xffffffffu;
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) v = __dadd_rn(v, __shfl_xor_sync(full, v, o));
    return quad_sum(v);
}

// jacobi_quad with one column per lane over 2^LC lanes and the two row pairs
// of a round in the halves of lane bit LC: (yp, yq) the half's rows, (zp, zq)
// their accumulated rotations.  Between rounds the first half's second row
// changes places with the other half's first, second, first row; after the
// last round the halves hold the rows 0, 1 and 2, 3 again.
template <int LC>
__device__ __forceinline__ void jacobi_warp(double &yp, double &yq, double &zp, double &zq, int lane)
{
    const unsigned full = 0xffffffffu;
    const bool second = (lane >> LC) & 1;
#pragma unroll 1
    for (int sweep = 0; sweep < 40; sweep++) {
        double al = row_dot_warp<LC>(yp, yp, lane), be = row_dot_warp<LC>(yq, yq, lane);
        bool any = false;
#pragma unroll
        for (int round = 0; round < 3; round++) {
            const double ga = row_dot_warp<LC>(yp, yq, lane);
            const bool rot = jac_needed64(al, be, ga);
            if (rot) {
                any = true;
                double th, sn;
                jac_shears64(al, be, ga, th, sn);
                yp = fma(-th, yq, yp);
                zp = fma(-th, zq, zp);
                yq = fma(sn, yp, yq);
                zq = fma(sn, zp, zq);
                yp = fma(-th, yq, yp);
                zp = fma(-th, zq, zp);
            }
            const bool first = second && round != 1;   // the row that leaves: the second, or this half's first
            const double y = __shfl_xor_sync(full, first ? yp : yq, 1 << LC);
            const double z = __shfl_xor_sync(full, first ? zp : zq, 1 << LC);
            const double n = __shfl_xor_sync(full, first ? al : be, 1 << LC);
            if (first && round == 2) {
                yp = yq;
                zp = zq;
                al = be;
                yq = y;
                zq = z;
                be = n;
            } else if (first) {
                yp = y;
                zp = z;
                al = n;
            } else {
                yq = y;
                zq = z;
                be = n;
            }
        }
        if (!__any_sync(full, any)) break;
    }
}

// singular values of the half's two rows, their reciprocals (0 for a zero
// row) and their places among the four in descending order
template <int LC>
__device__ __forceinline__ void svd_place_warp(double yp, double yq, double &sp, double &sq, double &ip, double &iq,
                                               int &pp, int &pq, int lane)
{
    const unsigned full = 0xffffffffu;
    const bool second = (lane >> LC) & 1;
    const double np = row_dot_warp<LC>(yp, yp, lane), nq = row_dot_warp<LC>(yq, yq, lane);
    // one root per lane (its lowest bit: the row), passed to the other
    const double nm = (lane & 1) ? nq : np, im = nm > 1e-290 ? rsqrt64(nm) : 0.0, sm = nm * im;
    const double io = __shfl_xor_sync(full, im, 1), so = __shfl_xor_sync(full, sm, 1);
    sp = (lane & 1) ? so : sm;
    sq = (lane & 1) ? sm : so;
    ip = (lane & 1) ? io : im;
    iq = (lane & 1) ? im : io;
    // (non-negative: ordered as their bits; equal ones in row order)
    const long long a = __double_as_longlong(sp), b = __double_as_longlong(sq);
    const long long c = __shfl_xor_sync(full, a, 1 << LC), d = __shfl_xor_sync(full, b, 1 << LC);
    pp = (b > a) + (c > a || (second && c == a)) + (d > a || (second && d == a));
    pq = (a >= b) + (c > b || (second && c == b)) + (d > b || (second && d == b));
}

__global__ void __launch_bounds__(32 * E64W_WARPS) k_estimate_f64w(GsProblem P, int level,
                                                                   const double *__restrict__ A, int64_t n,
                                                                   const uint64_t *parents, const uint8_t *vmask,
                                                                   uint8_t *__restrict__ dec,
                                                                   double *__restrict__ bounds,
                                                                   const int32_t *__restrict__ list,
                                                                   const unsigned *nlist)
{
    __shared__ double s_V[E64W_WARPS][4][4][4], s_W[E64W_WARPS][4][4][4], s_u[E64W_WARPS][4][4];
    __shared__ double s_s[E64W_WARPS][4], s_d[E64W_WARPS][4][4], s_sd[E64W_WARPS][4][4];
    const unsigned full = 0xffffffffu;
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
    const int64_t cnt = list ? (int64_t)*nlist : n;
    if (cnt > E64W_MAX) return;   // k_estimate_f64 takes them
    const int64_t t = (int64_t)blockIdx.x * E64W_WARPS + wl;
    if (t >= cnt) return;
    const int64_t q = list ? (int64_t)list[t] : t;
    const Octet oc = octet_of(P, level, parents, vmask, q >> 3);
    if (!((oc.vmask >> (q & 7)) & 1)) {
        if (lane == 0) dec[q] = DEC_INVALID;
        return;
    }
    const double *a = A + q * 64;
    // column (lane & 15) of the unfolding; the half's first row pair
    const int col = lane & 15, h = lane >> 4;
    double yp = a[32 * h + col], yq = a[32 * h + 16 + col], zp = 2 * h == col, zq = 2 * h + 1 == col;
    const double both = __dadd_rn(fabs(yp), fabs(yq));
    const double high = entry_sum_warp(h || (col >> 2) >= 2 || (col & 3) >= 2 ? both : 0.0);
    const double tot = entry_sum_warp(both);
    double b[6] = {0, 0, 0, high, 0, 0}, rrel = 1e30;
    if (tot != 0.0) {
        double sp, sq, ip, iq, to, back;
        int pp, pq;
        const bool scaled = svd_scale64(tot, to, back);
        if (scaled) {
            yp *= to;
            yq *= to;
        }
        jacobi_warp<4>(yp, yq, zp, zq, lane);
        svd_place_warp<4>(yp, yq, sp, sq, ip, iq, pp, pq, lane);
        s_V[wl][pp][col >> 2][col & 3] = yp * ip;
        s_V[wl][pq][col >> 2][col & 3] = yq * iq;
        if (col < 4) {
            s_u[wl][pp][col] = zp;
            s_u[wl][pq][col] = zq;
            s_s[wl][pp] = sp;
            s_s[wl][pq] = sq;
        }
        __syncwarp();
        const double s[4] = {s_s[wl][0], s_s[wl][1], s_s[wl][2], s_s[wl][3]};
        double rm;
        const int jr = rank99(s, rm);
        rrel = rm / (s[0] + s[1] + s[2] + s[3]);
        // inner SVDs: lanes 8 i .. 8 i + 7 take V_i (its row pairs in lane bit 2)
        const int i = lane >> 3, g = (lane >> 2) & 1, l = lane & 3;
        double vp = i < jr ? s_V[wl][i][2 * g][l] : 0.0, vq = i < jr ? s_V[wl][i][2 * g + 1][l] : 0.0;
        double wp = 2 * g == l, wq = 2 * g + 1 == l;
        jacobi_warp<2>(vp, vq, wp, wq, lane);
        svd_place_warp<2>(vp, vq, sp, sq, ip, iq, pp, pq, lane);
        __syncwarp();
        s_V[wl][i][pp][l] = vp * ip;
        s_V[wl][i][pq][l] = vq * iq;
        s_W[wl][i][pp][l] = wp;
        s_W[wl][i][pq][l] = wq;
        s_d[wl][i][pp] = sp;
        s_d[wl][i][pq] = sq;
        __syncwarp();
        const double d[4] = {s_d[wl][i][0], s_d[wl][i][1], s_d[wl][i][2], s_d[wl][i][3]};
        double rmi;
        const int ji = i < jr ? rank99(d, rmi) : 0;
        double rri = i < jr ? rmi / (d[0] + d[1] + d[2] + d[3]) : 1e30;
        int inner = ji;
#pragma unroll
        for (int o = 8; o < 32; o <<= 1) {
            rri = fmin(rri, __shfl_xor_sync(full, rri, o));
            inner += __shfl_xor_sync(full, inner, o);
        }
        rrel = fmin(rrel, rri);
        const double si = s_s[wl][i], dl = s_d[wl][i][l];
        if (g == 0) s_sd[wl][i][l] = l < ji ? si * dl : 0.0;
        __syncwarp();
        // 1-D ranges: lane (i, 0, k) of w_ik, lane (i, 1, k) of V_ik, then of u_i
        double cf[4], lo, hi, lx, hx;
#pragma unroll
        for (int k = 0; k < 4; k++) cf[k] = g ? s_V[wl][i][l][k] : s_W[wl][i][l][k];
        cubic_range64(cf, lo, hi);
#pragma unroll
        for (int k = 0; k < 4; k++) cf[k] = s_u[wl][i][k];
        cubic_range64(cf, lx, hx);
        const double lo2 = __shfl_xor_sync(full, lo, 4), hi2 = __shfl_xor_sync(full, hi, 4);
        double mn, mx;
        product_range(lo, hi, lo2, hi2, mn, mx);
        const double Myz = quad_sum(l < ji ? __dmul_rn(dl, mx) : 0.0);
        const double myz = quad_sum(l < ji ? __dmul_rn(dl, mn) : 0.0);
        product_range(lx, hx, myz, Myz, mn, mx);
        double M = 0.0, m = 0.0;
        for (int ii = 0; ii < jr; ii++) {
            M = fma(s[ii], __shfl_sync(full, mx, 8 * ii), M);
            m = fma(s[ii], __shfl_sync(full, mn, 8 * ii), m);
        }
        // residual: the lane's entries of its first layout
        double r0 = a[32 * h + col], r1 = a[32 * h + 16 + col];
        if (scaled) {
            r0 *= to;
            r1 *= to;
        }
        for (int ii = 0; ii < jr; ii++)
            for (int k = 0; k < 4; k++) {
                const double sd = s_sd[wl][ii][k];
                if (sd == 0.0) break;   // past the kept terms
                const double xw = sd * s_V[wl][ii][k][col & 3] * s_W[wl][ii][k][col >> 2];
                r0 = fma(-s_u[wl][ii][2 * h], xw, r0);
                r1 = fma(-s_u[wl][ii][2 * h + 1], xw, r1);
            }
        const double sr = entry_sum_warp(__dadd_rn(fabs(r0), fabs(r1)));
        b[0] = (m - sr) * back;
        b[1] = (M + sr) * back;
        b[2] = sr * back;
        b[4] = (double)jr;
        b[5] = (double)inner;
    }
    if (lane == 0) finish_f64(P, level, q, a, b, rrel, dec, bounds);
}

// the FP64 estimate of n cubes, or of the *nlist listed ones (at most n); the
// number decides on the device which of the two kernels works
static void launch_estimate_f64(const GsProblem &P, int level, const double *d_A, int64_t n, const uint64_t *d_parents,
                                const uint8_t *d_vmask, uint8_t *d_dec, double *d_bounds, const int32_t *list,
                                const unsigned *nlist, cudaStream_t st)
{
    if (list || n <= E64W_MAX) {
        const int64_t m = n < E64W_MAX ? n : E64W_MAX;
        GS_LAUNCH(k_estimate_f64w, (unsigned)((m + E64W_WARPS - 1) / E64W_WARPS), 32 * E64W_WARPS, 0, st)(
            P, level, d_A, n, d_parents, d_vmask, d_dec, d_bounds, list, nlist);
    }
    if (n > E64W_MAX)
        GS_LAUNCH(k_estimate_f64, (unsigned)((n + 31) / 32), 128, 0, st)(P, level, d_A, n, d_parents, d_vmask, d_dec,
                                                                        d_bounds, list, nlist);
}

// FP64 first pass (default decision order and norm, no bounds wanted):
// invalid cubes and cubes whose corner values of P~ straddle c by more than
// the rounding of those sums (1e-12 sum|A|) are decided here; the FP64 bounds
// enclose P~ up to rounding, so the SVD estimate would keep them too, and
// the precision sum is taken in the same order as there.  The rest go to a
// list for the SVD estimate.
__global__ void __launch_bounds__(256) k_estimate_pre64(GsProblem P, int level, const double *__restrict__ A, int64_t n,
                                                        const uint64_t *parents, const uint8_t *vmask,
                                                        uint8_t *__restrict__ dec, int32_t *__restrict__ list,
                                                        unsigned *nlist)
{
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    bool slow = false;
    if (q < n) {
        Octet oc = octet_of(P, level, parents, vmask, q >> 3);
        if (!((oc.vmask >> (q & 7)) & 1)) {
            dec[q] = DEC_INVALID;
        } else {
            double a[64];
            double tot = 0.0, high = 0.0;
#pragma unroll
            for (int t = 0; t < 64; t++) {
                a[t] = A[q * 64 + t];
                tot += fabs(a[t]);
                if ((t >> 4) >= 2 || ((t >> 2) & 3) >= 2 || (t & 3) >= 2) high += fabs(a[t]);
            }
            double lo, hi;
            corner_range<double>(a, lo, hi);
            const double cm = 1e-12 * tot;
            if (tot == 0.0) {
                // no atom reaches the cube: the full estimate discards it
                dec[q] = DEC_DISCARD;
            } else if (hi - P.c > cm && P.c - lo > cm) {
                dec[q] = (uint8_t)(high <= P.precision ? DEC_ACCEPT : (level >= P.max_depth ? DEC_FORCED : DEC_SPLIT));
                if (P.near && fabs(P.precision - high) < GS_NEAR_REL * (P.precision + high))
                    atomicAdd(&P.near[1], 1ull);
            } else {
                // the bounds' own margins (near_threshold) and the rounding of
                // these sums stay far below 1e-8 (c + sum|A|)
                double mn, mx;
                trilinear_range<double>(a, high, mn, mx);
                const double room = fmax(P.c - mx, mn - P.c) - 1e-8 * (P.c + tot);
                slow = true;
                if (room > 1e-150 && fabs(a[0]) > 1e-3 * tot &&
                    RANK_ONE_SLOPE * RANK_ONE_SLOPE * rank_one_dist2<double>(a) < room * room) {
                    dec[q] = DEC_DISCARD;
                    slow = false;
                }
            }
        }
    }
    const unsigned bal = __ballot_sync(0xffffffffu, slow);
    if (!bal) return;
    const unsigned lane = threadIdx.x & 31;
    unsigned wb = 0;
    if (lane == 0) wb = atomicAdd(nlist, (unsigned)__popc(bal));
    wb = __shfl_sync(0xffffffffu, wb, 0);
    if (slow) list[wb + __popc(bal & ((1u << lane) - 1u))] = (int32_t)q;
}

int gs_estimate_f64(const GsProblem &P, int level, const double *d_A, int64_t n_cubes, const uint64_t *d_parents,
                    const uint8_t *d_vmask, uint8_t *d_dec, double *d_bounds, cudaStream_t st)
{
    if (n_cubes <= 0) return GS_OK;
    if (!d_bounds && P.order == GS_ORDER_BOUNDS_FIRST && P.norm == GS_NORM_SUM && n_cubes < ((int64_t)1 << 31)) {
        int32_t *list = nullptr;
        unsigned *nlist = nullptr;
        int rc = gs_alloc((void **)&list, sizeof(int32_t) * (size_t)n_cubes, st);
        if (!rc) rc = gs_alloc((void **)&nlist, sizeof(unsigned), st);
        if (rc) { gs_free(list, st); return rc; }
        GS_CHECK(cudaMemsetAsync(nlist, 0, sizeof(unsigned), st));
        GS_LAUNCH(k_estimate_pre64, (unsigned)((n_cubes + 255) / 256), 256, 0, st)(P, level, d_A, n_cubes, d_parents,
                                                                                d_vmask, d_dec, list, nlist);
        launch_estimate_f64(P, level, d_A, n_cubes, d_parents, d_vmask, d_dec, nullptr, list, nlist, st);
        gs_free(list, st);
        gs_free(nlist, st);
        GS_CHECK(cudaGetLastError());
        return GS_OK;
    }
    launch_estimate_f64(P, level, d_A, n_cubes, d_parents, d_vmask, d_dec, d_bounds, nullptr, nullptr, st);
    GS_CHECK(cudaGetLastError());
    return GS_OK;
}

// ---------------------------------------------------------------- re-expansion
// child tensors from the parents' (one thread per child): the parent's
// polynomial re-expanded on the child box, axis by axis
__global__ void k_reexpand(const double *__restrict__ Apar, int64_t n_oct, double *__restrict__ A_out)
{
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n_oct * 8) return;
    const int c = (int)(t & 7), hx = c & 1, hy = (c >> 1) & 1, hz = c >> 2;
    const double *P = Apar + (t >> 3) * 64;
    double B[64], C[64];
    // along x (first index)
    for (int p = 0; p < 4; p++)
        for (int kl = 0; kl < 16; kl++) {
            double acc = 0.0;
            for (int j = 0; j < 4; j++) acc = fma(c_reexp[hx][p][j], P[16 * j + kl], acc);
            B[16 * p + kl] = acc;
        }
    // along y
    for (int p = 0; p < 4; p++)
        for (int q = 0; q < 4; q++)
            for (int l = 0; l < 4; l++) {
                double acc = 0.0;
                for (int k = 0; k < 4; k++) acc = fma(c_reexp[hy][q][k], B[16 * p + 4 * k + l], acc);
                C[16 * p + 4 * q + l] = acc;
            }
    // along z
    double *out = A_out + t * 64;
    for (int pq = 0; pq < 16; pq++)
        for (int r = 0; r < 4; r++) {
            double acc = 0.0;
            for (int l = 0; l < 4; l++) acc = fma(c_reexp[hz][r][l], C[4 * pq + l], acc);
            out[4 * pq + r] = acc;
        }
}

int gs_reexpand(const double *d_Apar, int64_t n_oct, double *d_A, cudaStream_t st)
{
    if (n_oct <= 0) return GS_OK;
    GS_LAUNCH(k_reexpand, (unsigned)((n_oct * 8 + 127) / 128), 128, 0, st)(d_Apar, n_oct, d_A);
    GS_CHECK(cudaGetLastError());
    return GS_OK;
}

// tensors of the split cubes, in the order of the next level's parents
__global__ void k_split_tensors(const uint8_t *__restrict__ dec, int64_t n, const int64_t *__restrict__ off,
                                const double *__restrict__ A, double *__restrict__ Anext)
{
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n * 64) return;
    const int64_t q = t >> 6;
    if (dec[q] != DEC_SPLIT) return;
    Anext[(off[q] & 0xffffffffll) * 64 + (t & 63)] = A[t];
}

// ---------------------------------------------------------------- compaction
// packed[q] = [SPLIT] + [ACCEPT or FORCED] << 32; after an exclusive scan the
// low half is the cube's slot among the next level's parents, the high half
// its slot among the accepted cubes.  counters: examined, discarded,
// accepted, forced, split.
__global__ void __launch_bounds__(256) k_level_count(const uint8_t *__restrict__ dec, int64_t n,
                                                     int64_t *__restrict__ packed, unsigned long long *counters)
{
    // grid-stride; counts kept per thread and reduced once per block, so the
    // five global counters see one atomic per block
    unsigned cnt[5] = {0, 0, 0, 0, 0};
    for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < n; q += (int64_t)gridDim.x * blockDim.x) {
        unsigned d = dec[q];
        packed[q] = (int64_t)(d == DEC_SPLIT) | ((int64_t)(d == DEC_ACCEPT || d == DEC_FORCED) << 32);
        cnt[0] += d != DEC_INVALID;
        cnt[1] += d == DEC_DISCARD;
        cnt[2] += d == DEC_ACCEPT;
        cnt[3] += d == DEC_FORCED;
        cnt[4] += d == DEC_SPLIT;
    }
    __shared__ unsigned long long sh[5];
    if (threadIdx.x < 5) sh[threadIdx.x] = 0;
    __syncthreads();
    for (int k = 0; k < 5; k++) {
        unsigned v = cnt[k];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if ((threadIdx.x & 31) == 0 && v) atomicAdd(&sh[k], (unsigned long long)v);
    }
    __syncthreads();
    if (threadIdx.x < 5 && sh[threadIdx.x]) atomicAdd(&counters[threadIdx.x], sh[threadIdx.x]);
}

// mol (nullable, the batched form): the octets' molecules, passed on to the
// children (next_mol) and the accepted cubes (acc_mol)
__global__ void k_level_emit(GsProblem P, int level, const uint64_t *parents, const uint8_t *vmask,
                             const uint8_t *__restrict__ dec, int64_t n, const int64_t *__restrict__ off,
                             uint64_t *__restrict__ next, uint64_t *__restrict__ acc, const int32_t *__restrict__ mol,
                             int32_t *__restrict__ next_mol, int32_t *__restrict__ acc_mol)
{
    int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    unsigned d = dec[q];
    if (d != DEC_SPLIT && d != DEC_ACCEPT && d != DEC_FORCED) return;
    Octet oc = octet_of(P, level, parents, vmask, q >> 3);
    int c = (int)(q & 7);
    uint64_t key = gk_make(2 * oc.I + (c & 1), 2 * oc.J + ((c >> 1) & 1), 2 * oc.K + (c >> 2), GT_CUBE, (unsigned)level);
    int64_t o = off[q];
    if (d == DEC_SPLIT) {
        next[o & 0xffffffffll] = key;
        if (mol) next_mol[o & 0xffffffffll] = mol[q >> 3];
    } else {
        acc[o >> 32] = key;
        if (mol) acc_mol[o >> 32] = mol[q >> 3];
    }
}

int gs_level_compact(const GsProblem &P, int level, const uint64_t *d_parents, const uint8_t *d_vmask, int64_t n_oct,
                     const uint8_t *d_dec, uint64_t **d_next, int64_t *n_next, uint64_t *d_acc_base,
                     int64_t acc_cap, int64_t *n_acc, unsigned long long *d_counters, cudaStream_t st,
                     const double *d_A, double **d_nextA, const int32_t *d_mol, int32_t **d_next_mol,
                     int32_t *d_acc_mol)
{
    if (d_nextA) *d_nextA = nullptr;
    if (d_next_mol) *d_next_mol = nullptr;
    int64_t n = n_oct * 8;
    *d_next = nullptr; *n_next = 0; *n_acc = 0;
    if (n <= 0) return GS_OK;
    int64_t *packed = nullptr, *tot = nullptr;
    int rc = gs_alloc((void **)&packed, sizeof(int64_t) * (size_t)(n + 1), st);
    if (!rc) rc = gs_alloc((void **)&tot, sizeof(int64_t), st);
    if (rc) { gs_free(packed, st); return rc; }
    cudaMemsetAsync(packed + n, 0, sizeof(int64_t), st);
    {
        int64_t nb = (n + 255) / 256;
        GS_LAUNCH(k_level_count, (unsigned)(nb < 152 * 16 ? nb : 152 * 16), 256, 0, st)(d_dec, n, packed, d_counters);
    }
    rc = gs_scan_i64(packed, n + 1, tot, st);
    int64_t h = 0;
    if (!rc) {
        cudaError_t e = cudaMemcpyAsync(&h, tot, sizeof(int64_t), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = gs_sync(st);
        if (e != cudaSuccess) rc = gs_fail_cuda(e, "level counts", __FILE__, __LINE__);
    }
    int64_t ns = h & 0xffffffffll, na = h >> 32;
    if (!rc && na > acc_cap) rc = gs_fail(GS_ERR_CAPACITY, "accepted-cube buffer too small");
    if (!rc && ns > 0) rc = gs_alloc((void **)d_next, sizeof(uint64_t) * (size_t)ns, st);
    if (!rc && ns > 0 && d_mol) rc = gs_alloc((void **)d_next_mol, sizeof(int32_t) * (size_t)ns, st);
    if (!rc) GS_LAUNCH(k_level_emit, (unsigned)((n + 255) / 256), 256, 0, st)(P, level, d_parents, d_vmask, d_dec, n, packed,
                                                                      *d_next, d_acc_base, d_mol,
                                                                      d_mol ? *d_next_mol : nullptr, d_acc_mol);
    if (!rc && d_A && d_nextA && ns > 0) {
        rc = gs_alloc((void **)d_nextA, sizeof(double) * 64 * (size_t)ns, st);
        if (!rc)
            GS_LAUNCH(k_split_tensors, (unsigned)((n * 64 + 255) / 256), 256, 0, st)(d_dec, n, packed, d_A, *d_nextA);
    }
    gs_free(packed, st); gs_free(tot, st);
    if (rc) return rc;
    GS_CHECK(cudaGetLastError());
    *n_next = ns;
    *n_acc = na;
    return GS_OK;
}

// explicit keys of the root blocks (2x2x2 root cubes), x fastest
__global__ void k_root_blocks(int64_t bx, int64_t by, int64_t n, uint64_t *keys)
{
    int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= n) return;
    keys[o] = gk_make(o % bx, (o / bx) % by, o / (bx * by), GT_CUBE, 0);
}

int gs_root_blocks(const GsProblem &P, uint64_t **d_keys, int64_t *n, cudaStream_t st)
{
    int64_t bx = (P.nroot[0] + 1) / 2, by = (P.nroot[1] + 1) / 2, bz = (P.nroot[2] + 1) / 2;
    *n = bx * by * bz;
    int rc = gs_alloc((void **)d_keys, sizeof(uint64_t) * (size_t)*n, st);
    if (rc) return rc;
    GS_LAUNCH(k_root_blocks, (unsigned)((*n + 255) / 256), 256, 0, st)(bx, by, *n, *d_keys);
    GS_CHECK(cudaGetLastError());
    return GS_OK;
}

// ================================================================ mixed precision
// FP32 accumulation.  Atom centres and lattice coordinates are taken relative
// to the origin as two-float sums, so differences x - e keep ~1e-7 A; the
// 1-D factors use gs_ex2; each lane sums 8 atoms plainly and folds the batch
// into a Kahan-compensated accumulator.  Per cube it also sums
// w * Fx * Fy * Fz (F = the largest value of the atom's 1-D factor on the
// cube's interval), an upper bound of every term's size from which the
// error band of the FP32 tensor is derived.
// Per queued atom the coefficient lane writes the products the update needs:
// WXY[cy][cx][j][k] = w X_cx[j] Y_cy[k] (64) and Z[cz][l] with each value
// twice (16); the update of lane (child, j) is then three 16-byte loads and 8
// paired FMA (f32x2) per atom: the pairs run over k = (0,1) and (2,3) against
// (Z[l], Z[l]).  The eight lanes of a quarter warp read eight consecutive
// 16-byte words; the record stride (21 words of 16 bytes) spreads the
// coefficient lanes' stores over all banks.  The records of the atoms that
// reach all eight children come first, so that three quarters of the updates
// need no mask.  Per child the sum of w Fx Fy Fz is kept by the coefficient
// lanes (one addition per atom and child there, where the update lanes spent
// four instructions per atom on it) and reduced once per octet.  20,000
// atoms, finest level: 1.35 -> 1.15 ms, issue slots 60% busy, shared-memory
// pipe 64%; five blocks per SM at 96 registers spill (1.46 ms), three at 168
// hide less latency (1.21 ms).
#define ACF_WXY 0
#define ACF_Z 64
#define ACF_MASK 80
#define ACF_STRIDE 84

// one axis, FP32: the coefficients of both child intervals (cf[h]) and F[h],
// the largest value of the factor on interval h, from the lattice ends as hi
// + lo floats and the atom's offset likewise; D2 = -D log2(e)
template <int GV, int NQ>
struct Quad32 {
    __device__ __forceinline__ void axis(const float *eh, const float *el, float ah, float al, float hh, float D2,
                                         float2 (&cf)[4], float2 &F) const
    {
        float d[3], f[3], a[2][4], g[2];
#pragma unroll
        for (int t = 0; t < 3; t++) {
            d[t] = (eh[t] - ah) + (el[t] - al);   // e_t - x
            f[t] = gs_ex2(D2 * d[t] * d[t]);
        }
#pragma unroll
        for (int h = 0; h < 2; h++) {
            const float m = d[h] + hh;   // interval centre - x
            float a0 = 0.f, a1 = 0.f;
#pragma unroll
            for (int k = 0; k < NQ; k++) {
                float dk = fmaf(hh, c_gq_tf[GV][k], m);
                float fk = gs_ex2(D2 * dk * dk);
                a0 = fmaf(c_gq_Wf[GV][k][0], fk, a0);
                a1 = fmaf(c_gq_Wf[GV][k][1], fk, a1);
            }
            a[h][0] = a0;
            a[h][1] = a1;
            a[h][2] = 0.5f * (f[h] + f[h + 1]) - a0;
            a[h][3] = 0.5f * (f[h + 1] - f[h]) - a1;
            g[h] = d[h] <= 0.f && d[h + 1] >= 0.f ? 1.f : fmaxf(f[h], f[h + 1]);
        }
#pragma unroll
        for (int q = 0; q < 4; q++) cf[q] = make_float2(a[0][q], a[1][q]);
        F = make_float2(g[0], g[1]);
    }
};
template <int K>
struct Series32 {
    float2 c[4][K];   // each coefficient twice
    float kappa;
    __device__ __forceinline__ void axis(const float *eh, const float *el, float ah, float al, float hh, float D2,
                                         float2 (&cf)[4], float2 &F) const
    {
        // one exponential stands for the whole interval, so its argument
        // -D m^2 is formed with the rounding errors of m (its low part l), of
        // m^2 and of the product: E = 2^g (1 + ln 2 r), r the sum of what g
        // lacks
        const float2 one = make_float2(-1.f, -1.f), DD = make_float2(D2, D2), hp = make_float2(-hh, hh);
        const float dh = eh[1] - ah, dl = el[1] - al, d1 = dh + dl, dr = dl - (d1 - dh);   // e_1 - x
        const float2 d = make_float2(d1, d1), m = __fadd2_rn(d, hp);
        const float2 l = __fadd2_rn(__ffma2_rn(__ffma2_rn(d, one, m), one, hp), make_float2(dr, dr));
        const float2 mu = __fmul2_rn(make_float2(kappa, kappa), m), s = __fmul2_rn(mu, mu);
        const float2 p2 = __fmul2_rn(m, m), g = __fmul2_rn(DD, p2);
        const float2 e = __ffma2_rn(__fadd2_rn(m, m), l, __ffma2_rn(m, m, make_float2(-p2.x, -p2.y)));
        const float2 r = __ffma2_rn(DD, e, __ffma2_rn(DD, p2, make_float2(-g.x, -g.y)));
        float2 E = make_float2(gs_ex2(g.x), gs_ex2(g.y));
        E = __ffma2_rn(E, __fmul2_rn(r, make_float2(0.69314718f, 0.69314718f)), E);
        const float2 o = __fmul2_rn(mu, E);
#pragma unroll
        for (int q = 0; q < 4; q++) {
            float2 p = c[q][K - 1];
#pragma unroll
            for (int k = K - 2; k >= 0; k--) p = __ffma2_rn(p, s, c[q][k]);
            cf[q] = __fmul2_rn(p, (q & 1) ? o : E);
        }
        // 1 inside the interval; outside, the value at the nearer end, which
        // the corrected series takes there: a0 + a2 +- (a1 + a3)
        const float2 u = __fadd2_rn(cf[0], cf[2]), v = __fadd2_rn(cf[1], cf[3]);
        F.x = fabsf(m.x) <= hh ? 1.f : u.x + fabsf(v.x);
        F.y = fabsf(m.y) <= hh ? 1.f : u.y + fabsf(v.y);
    }
};

template <class C, bool BATCH>
__global__ void __launch_bounds__(32 * ACC_WARPS, 4) k_accum_f32(const __grid_constant__ GsProblem P0, int level,
                                                                  const uint64_t *parents, const uint8_t *vmask,
                                                                  int64_t n_oct, float hf, float ctol, int lat_exact,
                                                                  const __grid_constant__ C coef,
                                                                  float *__restrict__ A_out,
                                                                  float *__restrict__ E_out,
                                                                  unsigned long long *pairs,
                                                                  unsigned long long *atom_octets,
                                                                  const GsProblem *__restrict__ probs,
                                                                  const int32_t *__restrict__ mol)
{
    unsigned long long my_pairs = 0, my_atoms = 0;
    __shared__ __align__(16) float s_cf[ACC_WARPS][32][ACF_STRIDE];
    __shared__ int s_qi[ACC_WARPS][ACC_Q];
    __shared__ uint8_t s_qm[ACC_WARPS][ACC_Q];
    const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5;
    const unsigned full = 0xffffffffu;
    const unsigned below = (1u << lane) - 1u;
    const int c = lane >> 2, j = lane & 3;
    const int cx = c & 1, cy = (c >> 1) & 1, cz = c >> 2;
    const int oWXY = ACF_WXY + ((cy * 2 + cx) * 4 + j) * 4, oZ = ACF_Z + 8 * cz;
    const float nDl2e = (float)(-P0.D * 1.4426950408889634);
    const float hh = 0.5f * hf;
    for (int64_t o = (int64_t)blockIdx.x * ACC_WARPS + wl; o < n_oct; o += (int64_t)gridDim.x * ACC_WARPS) {
        const GsProblem &P = BATCH ? probs[mol[o]] : P0;
        Octet q = octet_of(P, level, parents, vmask, o);
        int64_t base[3] = {2 * q.I, 2 * q.J, 2 * q.K};
        // interval ends relative to the origin as hi + lo floats; when the
        // lattice spacing has few mantissa bits the products are exact in FP32
        float eh[3][3], el[3][3];
        for (int a = 0; a < 3; a++)
            for (int t = 0; t < 3; t++) {
                if (lat_exact) {
                    // indices < 2^18: convert through int32 (64-bit conversions are slow)
                    eh[a][t] = (float)(int)(base[a] + t) * hf;
                    el[a][t] = 0.f;
                } else {
                    double rel = gs_lat(P, a, base[a] + t, level) - P.origin[a];
                    eh[a][t] = (float)rel;
                    el[a][t] = (float)(rel - (double)eh[a][t]);
                }
            }
        // [kp][l] holds the entries (k, l) = (2 kp, l) and (2 kp + 1, l);
        // ncomp is the negated Kahan compensation
        float2 acc[2][4], ncomp[2][4];
#pragma unroll
        for (int kp = 0; kp < 2; kp++)
#pragma unroll
            for (int l = 0; l < 4; l++) acc[kp][l] = ncomp[kp][l] = make_float2(0.f, 0.f);
        float eb[8];   // sums of w Fx Fy Fz per child over the atoms whose coefficients this lane computes
#pragma unroll
        for (int k = 0; k < 8; k++) eb[k] = 0.f;
        int qn = 0;
        const uint8_t vm = q.vmask;

        // coefficients of the queued atoms (one lane per atom), then the
        // rank-one updates (lane = child, x index) in batches of 8 atoms, each
        // summed plainly and folded into the compensated sums
        auto process = [&](int nproc) {
            const bool on = lane < nproc;
            const unsigned mk = on ? s_qm[wl][lane] : 0u;
            const unsigned whole = __ballot_sync(full, mk == 0xFFu);
            const int nw = __popc(whole);
            if (on) {
                const int i = s_qi[wl][lane];
                float2 cf[3][4], F[3];
                coef.axis(eh[0], el[0], P.hx[i], P.lx[i], hh, nDl2e, cf[0], F[0]);
                coef.axis(eh[1], el[1], P.hy[i], P.ly[i], hh, nDl2e, cf[1], F[1]);
                coef.axis(eh[2], el[2], P.hz[i], P.lz[i], hh, nDl2e, cf[2], F[2]);
                const float w = P.fw[i];
                float *rec = s_cf[wl][mk == 0xFFu ? __popc(whole & below) : nw + __popc(~whole & below)];
                *reinterpret_cast<unsigned *>(rec + ACF_MASK) = mk;
#pragma unroll
                for (int jj = 0; jj < 4; jj++) {
                    const float2 wx = __fmul2_rn(make_float2(w, w), cf[0][jj]);
#pragma unroll
                    for (int x = 0; x < 2; x++)
#pragma unroll
                        for (int y = 0; y < 2; y++) {
                            const float wv = x ? wx.y : wx.x;
                            const float2 w2 = make_float2(wv, wv);
                            const float2 p01 = __fmul2_rn(w2, y ? make_float2(cf[1][0].y, cf[1][1].y)
                                                                : make_float2(cf[1][0].x, cf[1][1].x));
                            const float2 p23 = __fmul2_rn(w2, y ? make_float2(cf[1][2].y, cf[1][3].y)
                                                                : make_float2(cf[1][2].x, cf[1][3].x));
                            *reinterpret_cast<float4 *>(rec + ACF_WXY + ((y * 2 + x) * 4 + jj) * 4) =
                                make_float4(p01.x, p01.y, p23.x, p23.y);
                        }
                }
                *reinterpret_cast<float4 *>(rec + ACF_Z) = make_float4(cf[2][0].x, cf[2][0].x, cf[2][1].x, cf[2][1].x);
                *reinterpret_cast<float4 *>(rec + ACF_Z + 4) = make_float4(cf[2][2].x, cf[2][2].x, cf[2][3].x, cf[2][3].x);
                *reinterpret_cast<float4 *>(rec + ACF_Z + 8) = make_float4(cf[2][0].y, cf[2][0].y, cf[2][1].y, cf[2][1].y);
                *reinterpret_cast<float4 *>(rec + ACF_Z + 12) = make_float4(cf[2][2].y, cf[2][2].y, cf[2][3].y, cf[2][3].y);
                const float2 wf = __fmul2_rn(make_float2(w, w), F[0]);
                const float2 f0 = __fmul2_rn(wf, make_float2(F[1].x, F[1].x)), f1 = __fmul2_rn(wf, make_float2(F[1].y, F[1].y));
#pragma unroll
                for (int cc = 0; cc < 8; cc++) {
                    const float2 ff = (cc & 2) ? f1 : f0;
                    const float t = ((cc & 1) ? ff.y : ff.x) * ((cc & 4) ? F[2].y : F[2].x);
                    if ((mk >> cc) & 1u) eb[cc] += t;
                }
            }
            __syncwarp();
            const float *rec0 = s_cf[wl][0];
#pragma unroll 1
            for (int t0 = 0; t0 < nproc; t0 += 8) {
                float2 part[2][4];
                if (t0 + 8 <= nw) {
#pragma unroll
                    for (int u = 0; u < 8; u++) {
                        const float *rec = rec0 + (t0 + u) * ACF_STRIDE;
                        const float4 xy = *reinterpret_cast<const float4 *>(rec + oWXY);
                        const float4 za = *reinterpret_cast<const float4 *>(rec + oZ);
                        const float4 zb = *reinterpret_cast<const float4 *>(rec + oZ + 4);
                        const float2 xk[2] = {make_float2(xy.x, xy.y), make_float2(xy.z, xy.w)};
                        const float2 zl[4] = {make_float2(za.x, za.y), make_float2(za.z, za.w), make_float2(zb.x, zb.y),
                                              make_float2(zb.z, zb.w)};
#pragma unroll
                        for (int kp = 0; kp < 2; kp++)
#pragma unroll
                            for (int l = 0; l < 4; l++)
                                part[kp][l] = u ? __ffma2_rn(xk[kp], zl[l], part[kp][l]) : __fmul2_rn(xk[kp], zl[l]);
                    }
                } else {
#pragma unroll
                    for (int kp = 0; kp < 2; kp++)
#pragma unroll
                        for (int l = 0; l < 4; l++) part[kp][l] = make_float2(0.f, 0.f);
                    const int te = t0 + 8 < nproc ? t0 + 8 : nproc;
#pragma unroll 1
                    for (int t = t0; t < te; t++) {
                        const float *rec = rec0 + t * ACF_STRIDE;
                        const unsigned mt = *reinterpret_cast<const unsigned *>(rec + ACF_MASK);
                        float4 xy = *reinterpret_cast<const float4 *>(rec + oWXY);
                        const float4 za = *reinterpret_cast<const float4 *>(rec + oZ);
                        const float4 zb = *reinterpret_cast<const float4 *>(rec + oZ + 4);
                        if (!((mt >> c) & 1u)) xy = make_float4(0.f, 0.f, 0.f, 0.f);   // not this lane's child
                        const float2 xk[2] = {make_float2(xy.x, xy.y), make_float2(xy.z, xy.w)};
                        const float2 zl[4] = {make_float2(za.x, za.y), make_float2(za.z, za.w), make_float2(zb.x, zb.y),
                                              make_float2(zb.z, zb.w)};
#pragma unroll
                        for (int kp = 0; kp < 2; kp++)
#pragma unroll
                            for (int l = 0; l < 4; l++) part[kp][l] = __ffma2_rn(xk[kp], zl[l], part[kp][l]);
                    }
                }
                // Kahan step y = part - comp, s = acc + y, comp = (s - acc) - y;
                // each subtraction is an FMA with -1, which rounds as it does
                const float2 m1 = make_float2(-1.f, -1.f);
#pragma unroll
                for (int kp = 0; kp < 2; kp++)
#pragma unroll
                    for (int l = 0; l < 4; l++) {
                        const float2 y = __fadd2_rn(part[kp][l], ncomp[kp][l]);
                        const float2 sm = __fadd2_rn(acc[kp][l], y);
                        const float2 t = __ffma2_rn(acc[kp][l], m1, sm);
                        ncomp[kp][l] = __ffma2_rn(t, m1, y);
                        acc[kp][l] = sm;
                    }
            }
            __syncwarp();
        };

        // membership of one candidate per lane (i < 0: none): FP32 box
        // distance with a relative margin, the exact FP64 test inside the
        // margin; members join the atom queue.  Per axis both gaps follow from
        // u = e_1 - x, whose rounding (1.3e-7 h with that of h) moves a squared
        // gap by up to 2.6e-7 h R <= 1.3e-7 h (R^2 + 1): the margin 1e-5 (R^2 + 1)
        // covers it up to h = 25 A, 4e-7 h (R^2 + 1) beyond.  t = d^2 - (R^2 -
        // tol) of a child is negative for a member, and as unsigned bits at
        // most those of 2 tol inside the margin
        auto filter = [&](int i) {
            unsigned m = 0;
            if (i >= 0) {
                const float ah[3] = {P.hx[i], P.hy[i], P.hz[i]}, al[3] = {P.lx[i], P.ly[i], P.lz[i]};
                float g2[3][2];
#pragma unroll
                for (int a = 0; a < 3; a++) {
                    const float u = (eh[a][1] - ah[a]) + (el[a][1] - al[a]);
                    const float g0 = fmaxf(fmaxf(u - hf, -u), 0.f), g1 = fmaxf(fmaxf(-u - hf, u), 0.f);
                    g2[a][0] = g0 * g0;
                    g2[a][1] = g1 * g1;
                }
                const float R2 = P.fR2[i];
                const float tol = ctol * R2 + ctol, lo = R2 - tol;
                unsigned tb[8], nmin = 0xffffffffu;
#pragma unroll
                for (int cc = 0; cc < 8; cc++) {
                    tb[cc] = __float_as_uint((g2[0][cc & 1] + g2[1][(cc >> 1) & 1]) - lo + g2[2][cc >> 2]);
                    m |= (tb[cc] >> 31) << cc;
                    nmin = min(nmin, tb[cc]);
                }
                const unsigned lim = __float_as_uint(2.f * tol);
                if (nmin <= lim) {
                    // near the cutoff sphere: the exact FP64 membership test
                    unsigned nearm = 0;
#pragma unroll
                    for (int cc = 0; cc < 8; cc++) nearm |= (tb[cc] <= lim ? 1u : 0u) << cc;
                    nearm &= vm;
                    while (nearm) {
                        const int cc = __ffs(nearm) - 1;
                        nearm &= nearm - 1;
                        double x = P.ax[i], y = P.ay[i], z = P.az[i];
                        int64_t ix = base[0] + (cc & 1), iy = base[1] + ((cc >> 1) & 1), iz = base[2] + (cc >> 2);
                        double dx = gs_axis_gap(gs_lat(P, 0, ix, level), gs_lat(P, 0, ix + 1, level), x);
                        double dy = gs_axis_gap(gs_lat(P, 1, iy, level), gs_lat(P, 1, iy + 1, level), y);
                        double dz = gs_axis_gap(gs_lat(P, 2, iz, level), gs_lat(P, 2, iz + 1, level), z);
                        double dd = __dadd_rn(__dadd_rn(__dmul_rn(dx, dx), __dmul_rn(dy, dy)), __dmul_rn(dz, dz));
                        if (dd <= P.aR2[i]) m |= 1u << cc;
                    }
                }
                m &= vm;
            }
            my_pairs += __popc(m);
            unsigned bal = __ballot_sync(full, m != 0);
            if (lane == 0) my_atoms += __popc(bal);
            int pos = qn + __popc(bal & below);
            if (m) { s_qi[wl][pos] = i; s_qm[wl][pos] = (uint8_t)m; }
            qn += __popc(bal);
            __syncwarp();
            if (qn >= 32) {
                process(32);
                int rest = qn - 32;
                int mi = 0; uint8_t mm = 0;
                if (lane < rest) { mi = s_qi[wl][32 + lane]; mm = s_qm[wl][32 + lane]; }
                __syncwarp();
                if (lane < rest) { s_qi[wl][lane] = mi; s_qm[wl][lane] = mm; }
                __syncwarp();
                qn = rest;
            }
        };

        if (vm) {
            float flo[3] = {eh[0][0], eh[1][0], eh[2][0]}, fhi[3] = {eh[0][2], eh[1][2], eh[2][2]};
            gs_warp_candidates(P, flo, fhi, lane, filter);
            if (qn > 0) process(qn);
        }
        float *dst = A_out + ((size_t)o * 8 + c) * 64 + 16 * j;
#pragma unroll
        for (int kp = 0; kp < 2; kp++) {
            float2 v[4];
#pragma unroll
            for (int l = 0; l < 4; l++) v[l] = __fadd2_rn(acc[kp][l], ncomp[kp][l]);   // acc - comp
            *reinterpret_cast<float4 *>(dst + 4 * (2 * kp)) = make_float4(v[0].x, v[1].x, v[2].x, v[3].x);
            *reinterpret_cast<float4 *>(dst + 4 * (2 * kp + 1)) = make_float4(v[0].y, v[1].y, v[2].y, v[3].y);
        }
        // the error sums over the lanes: each step halves the children a lane
        // keeps, so that lane 4 c + j ends with child c's
#pragma unroll
        for (int n = 4; n >= 1; n >>= 1) {
            const bool up = lane & (4 * n);
#pragma unroll
            for (int k = 0; k < n; k++) {
                const float r = __shfl_xor_sync(full, up ? eb[k] : eb[k + n], 4 * n);
                eb[k] = (up ? eb[k + n] : eb[k]) + r;
            }
        }
        eb[0] += __shfl_xor_sync(full, eb[0], 2);
        eb[0] += __shfl_xor_sync(full, eb[0], 1);
        if (j == 0) E_out[(size_t)o * 8 + c] = eb[0];
    }
    if (pairs) {
        for (int off = 16; off > 0; off >>= 1) my_pairs += __shfl_xor_sync(0xffffffffu, my_pairs, off);
        if (lane == 0 && my_pairs) atomicAdd(pairs, my_pairs);
    }
    if (atom_octets && lane == 0 && my_atoms) atomicAdd(atom_octets, my_atoms);
}

int gs_accum_f32(const GsProblem &P, int level, const uint64_t *d_parents, const uint8_t *d_vmask, int64_t n_oct,
                 float *d_A, float *d_err, unsigned long long *d_pairs, cudaStream_t st, cudaEvent_t *ev,
                 unsigned long long *d_atom_octets, const GsProblem *d_probs, const int32_t *d_mol)
{
    if (n_oct <= 0) return GS_OK;
    const double h = gs_h(P, level), hh = 0.5 * h;
    const float ctol = fmaxf(1e-5f, 4e-7f * (float)h);   // the membership margin (see the kernel's filter)
    if (ev) cudaEventRecord(ev[0], st);
    // grid shapes the tuner chooses from: up to 64, 16 or 4 blocks per SM
    // (each warp takes every grid-th octet; the sums do not depend on it)
    static const int64_t caps[3] = {152 * 64, 152 * 16, 152 * 4};
    auto run = [&](const char *name, auto coef) {
        using C = decltype(coef);
        return gs_tune_run(name, n_oct, 3, st, [&](int shape, unsigned long long *scratch) {
            int64_t g = (n_oct + ACC_WARPS - 1) / ACC_WARPS;
            if (g > caps[shape]) g = caps[shape];
            const unsigned grid = (unsigned)(g < 1 ? 1 : g);
            unsigned long long *pairs = scratch ? scratch : d_pairs;
            unsigned long long *aoct = scratch ? (d_atom_octets ? scratch + 1 : nullptr) : d_atom_octets;
            if (d_probs)
                GS_LAUNCH((k_accum_f32<C, true>), grid, 32 * ACC_WARPS, 0, st)(P, level, d_parents, d_vmask, n_oct,
                                                                             (float)h, ctol, P.lat_exact_f32, coef, d_A,
                                                                             d_err, pairs, aoct, d_probs, d_mol);
            else
                GS_LAUNCH((k_accum_f32<C, false>), grid, 32 * ACC_WARPS, 0, st)(P, level, d_parents, d_vmask, n_oct,
                                                                              (float)h, ctol, P.lat_exact_f32, coef, d_A,
                                                                              d_err, pairs, aoct, nullptr, nullptr);
        });
    };
    static const int Ks[] = {5, 6, 8, 11, 14};
    Series S;
    int K = 0;
    if (series_range32(P, hh)) K = series_coeffs(P.D, hh, P.pad, 2e-8, Ks, 5, &S);
    int rc;
#define GS_ACC32(K_)                                                                                          \
    case K_: {                                                                                                \
        Series32<K_> c;                                                                                       \
        c.kappa = (float)S.kappa;                                                                             \
        for (int q = 0; q < 4; q++)                                                                           \
            for (int k = 0; k < K_; k++) c.c[q][k] = make_float2((float)S.c[q][k], (float)S.c[q][k]);         \
        rc = run("k_accum_f32<series" #K_ ">", c);                                                            \
        break;                                                                                                \
    }
    switch (K) {
        GS_ACC32(5) GS_ACC32(6) GS_ACC32(8) GS_ACC32(11) GS_ACC32(14)
    default:
        if (gq_variant(P.D, hh, true) == 0) rc = run("k_accum_f32<nodes8>", Quad32<0, 8>());
        else rc = run("k_accum_f32<nodes16>", Quad32<1, 16>());
    }
#undef GS_ACC32
    if (rc) return rc;
    if (ev) cudaEventRecord(ev[1], st);
    GS_CHECK(cudaGetLastError());
    return GS_OK;
}

// FP32 estimate.  A decision is final when every margin it rests on exceeds
// the band the FP32 error of A and the FP32 estimate can move it by:
//   entry error      dA = MIXED_KAPPA * E + 1e-7 sum|A|   (E = sum w Fx Fy Fz;
//                    the largest observed |A32 - A64| / E is 7.7e-7)
//   bounds L, U      4 (dA + 1e-7 sum|A|)(1 + s), s = sigma_1 over the smallest
//                    gap between kept and neighbouring singular values (the
//                    singular vectors' sensitivity); about 9x the largest
//                    change observed between the FP32 and FP64 estimates
//   rank rules       a rule within 32 dA of its 99% threshold may flip and
//                    move terms between the main part and R; the decision is
//                    final when its margin also exceeds RANK_FLIP_ALLOW times
//                    the sum of the singular values; otherwise one such rule
//                    is settled by re-estimating under the flipped rank, more
//                    by FP64
//   precision sum    |d sum|high|| <= 64 dA + rounding (kept cubes only)
// Otherwise the cube is flagged and its octet is re-evaluated in FP64.  The
// debug mode (GS debug bit 0) re-runs every cube in FP64 and counts
// disagreements; the tests require zero.
#define MIXED_KAPPA 1.5e-6f

// Largest change of L or U, relative to the sum of the outer singular values
// S, when rank rules near their 99% thresholds flip.  A flipping rule moves
// terms whose singular values sum to at most ~1% of S (the rule sits at the
// threshold); per unit of singular value, a term adds at most 16 to the
// product bound (|u| <= sum|u_a| <= 2, sum d_k <= 2, |w z| <= 4) and at most 8
// to sum|R|.  Outer rules move <= 16 (0.011 S); inner rules of term i move
// <= 8 (0.011 sigma_i) sum_k d_k <= 16 (0.011 sigma_i), <= 16 (0.011 S) over
// all terms; together <= 0.36 S.
#define RANK_FLIP_ALLOW 0.4f

// Cubes whose corner values of P~ straddle c by more than the FP32 error of
// those sums are kept by the FP64 estimate whatever its SVD gives: L <= min P~
// and max P~ <= U hold for any factorisation, since R = A - A~ is taken
// exactly and the 1-D and product bounds are enclosures.  Their decision needs
// only the precision sum.  Returns false for the cubes that need the bounds.
__device__ __forceinline__ bool estimate_fast_f32(const GsProblem &P, int level, const float *__restrict__ A,
                                                  const float *__restrict__ E, int64_t q, const uint64_t *parents,
                                                  const uint8_t *vmask, uint8_t *__restrict__ dec,
                                                  uint8_t *__restrict__ flag, unsigned long long *why_cnt,
                                                  float *__restrict__ dbg)
{
    Octet oc = octet_of(P, level, parents, vmask, q >> 3);
    if (!((oc.vmask >> (q & 7)) & 1)) { dec[q] = DEC_INVALID; flag[q] = 0; return true; }
    float a[64];
    load_tensor_f32(A + q * 64, a);
    float tot = 0.f, high = 0.f;
#pragma unroll
    for (int t = 0; t < 64; t++) {
        tot += fabsf(a[t]);
        if ((t >> 4) >= 2 || ((t >> 2) & 3) >= 2 || (t & 3) >= 2) high += fabsf(a[t]);
    }
    if (tot == 0.f && E[q] == 0.f) {
        // no atom reaches the cube: P~ = 0 and the full estimate discards it
        // (zero bounds, no flag); common among the root cubes
        dec[q] = DEC_DISCARD;
        flag[q] = 0;
        if (why_cnt) atomicAdd(&why_cnt[10], 1ull);   // decided without the SVD
        if (dbg) {
            float *o = dbg + 6 * q;
            o[0] = o[1] = o[2] = o[3] = o[4] = 0.f;
            o[5] = 2.f;   // no SVD bounds: the band check skips the cube
        }
        return true;
    }
    const float c = (float)P.c, prec = (float)P.precision;
    const float dA = MIXED_KAPPA * E[q] + 1e-7f * tot;
    float lo, hi;
    corner_range<float>(a, lo, hi);
    // each corner sum moves by at most sum|dA_t| <= 64 dA, plus its own FP32
    // rounding (6 additions deep, < 4e-7 sum|A|)
    const float cm = 64.f * dA + 4e-6f * tot;
    if (!(hi - c > cm && c - lo > cm)) {
        // Discarded without the SVD (see trilinear_range): the FP64 tensor's
        // entries lie within dA, so its range within 64 dA and its distance
        // from the rank-one tensor within 8 dA of these, plus the FP32
        // rounding of the sums (below 4e-6 and 1e-6 sum|A|)
        float mn, mx;
        trilinear_range<float>(a, high, mn, mx);
        const float room = fmaxf(c - mx, mn - c) - cm - RANK_ONE_SLOPE * (8.f * dA + 1e-6f * tot);
        if (!(room > 1e-17f && fabsf(a[0]) > 1e-3f * tot &&
              1.0001f * (RANK_ONE_SLOPE * RANK_ONE_SLOPE) * rank_one_dist2<float>(a) < room * room))
            return false;
        if (why_cnt) atomicAdd(&why_cnt[10], 1ull);   // decided without the SVD
        if (dbg) {
            float *o = dbg + 6 * q;
            o[0] = lo; o[1] = hi; o[2] = 0.f; o[3] = dA; o[4] = tot;
            o[5] = 2.f;   // no SVD bounds: the band check skips the cube
        }
        dec[q] = DEC_DISCARD;
        flag[q] = 0;
        return true;
    }
    const int d = high <= prec ? DEC_ACCEPT : (level >= P.max_depth ? DEC_FORCED : DEC_SPLIT);
    if (why_cnt) atomicAdd(&why_cnt[10], 1ull);   // decided without the SVD
    const bool f = level < P.max_depth && fabsf(prec - high) <= 64.f * dA + 1e-6f * high + 1e-7f * tot;
    if (f && why_cnt) atomicAdd(&why_cnt[1], 1ull);
    if (dbg) {
        float *o = dbg + 6 * q;
        o[0] = lo; o[1] = hi; o[2] = 0.f; o[3] = dA; o[4] = tot;
        o[5] = 2.f;   // no SVD bounds: the band check skips the cube
    }
    dec[q] = (uint8_t)d;
    flag[q] = f ? 1 : 0;
    return true;
}

// the full FP32 estimate of one valid cube: two-level SVD bounds, rank rules
// and the bands below
__device__ __forceinline__ void estimate_full_f32(const GsProblem &P, int level, const float *__restrict__ A,
                                                  const float *__restrict__ E, int64_t q, uint8_t *__restrict__ dec,
                                                  uint8_t *__restrict__ flag, unsigned long long *why_cnt,
                                                  float *__restrict__ dbg, float *S)
{
    float tot = 0.f;
    {
        float a[64];
        load_tensor_f32(A + q * 64, a);
#pragma unroll
        for (int t = 0; t < 64; t++) tot += fabsf(a[t]);
    }
    float b[6], rm;
    float sens;
    RankNear rn;
    rn.m1 = rn.m2 = 1e30f; rn.who = -1; rn.alt = 0; rn.ssum = 0.f;
    estimate_bounds_sens(A + q * 64, S, b, rm, sens, 0, -1, 0, &rn);
    const float c = (float)P.c, prec = (float)P.precision;
    int d = decide<float>(b, c, prec, level, P.max_depth);
    float dA = MIXED_KAPPA * E[q] + 1e-7f * tot;
    bool f = false;
    int why = 0, alt = 0;
    if (tot > 0.f) {
        // calibrated: the largest |dL|, |dU| seen between the FP32 and FP64
        // estimates (debug mode, chain and globular molecules) is 0.85 of
        // (dA + 1e-7 sum|A|)(1 + s); the band takes 4 of it
        const float bBase = 4.f * (dA + 1e-7f * tot) * (1.f + fminf(sens, 1e4f));
        float mc = fminf(fabsf(c - b[0]), fabsf(b[1] - c));
        bool keep = b[0] <= c && c <= b[1];
        const float near = 32.f * dA + 1e-5f * tot;
        if (mc <= bBase) {
            f = true;
            why = 1;
        } else if (rn.m1 <= near && mc > bBase + RANK_FLIP_ALLOW * rn.ssum) {
            // rank rules within their band may flip, but no flip can move L
            // or U across c (see RANK_FLIP_ALLOW)
        } else if (rn.m1 <= near) {
            // a rank rule within its band may flip.  With one such rule the
            // cube is re-estimated under the flipped rank (k_estimate_alt);
            // with more, FP64 decides.
            if (rn.m2 > near && rn.alt > 0) {
                alt = 0x80 | ((rn.who + 1) << 3) | rn.alt;
            } else {
                f = true;
                why = 1;
                if (why_cnt) atomicAdd(&why_cnt[5], 1ull);   // flagged through a rank rule
            }
        }
        if (!f && keep && level < P.max_depth && fabsf(prec - b[3]) <= 64.f * dA + 1e-6f * b[3] + 1e-7f * tot) {
            f = true;
            why = 2;
        }
        if (f) alt = 0;
    } else if (E[q] > 0.f) {
        f = true;  // an all-zero FP32 tensor with contributing atoms: let FP64 decide
        why = 3;
    }
    if (why && why_cnt) atomicAdd(&why_cnt[why - 1], 1ull);
    if (dbg) {
        float *o = dbg + 6 * q;
        o[0] = b[0]; o[1] = b[1]; o[2] = sens; o[3] = dA; o[4] = tot;
        o[5] = (tot > 0.f && rn.m1 <= 32.f * dA + 1e-5f * tot) ? 1.f : 0.f;
    }
    dec[q] = (uint8_t)d;
    flag[q] = f ? 1 : (uint8_t)alt;}

// first pass: invalid and straddling cubes are decided here (one light thread
// per cube); the others go to a list that the SVD estimate runs over in full
// warps
__global__ void __launch_bounds__(256) k_estimate_pre(GsProblem P, int level, const float *__restrict__ A,
                                                      const float *__restrict__ E, int64_t n, const uint64_t *parents,
                                                      const uint8_t *vmask, uint8_t *__restrict__ dec,
                                                      uint8_t *__restrict__ flag, unsigned long long *why_cnt,
                                                      float *__restrict__ dbg, int32_t *__restrict__ list,
                                                      unsigned *nlist)
{
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const bool slow = q < n && !estimate_fast_f32(P, level, A, E, q, parents, vmask, dec, flag, why_cnt, dbg);
    const unsigned bal = __ballot_sync(0xffffffffu, slow);
    if (!bal) return;
    const unsigned lane = threadIdx.x & 31;
    unsigned wb = 0;
    if (lane == 0) wb = atomicAdd(nlist, (unsigned)__popc(bal));
    wb = __shfl_sync(0xffffffffu, wb, 0);
    if (slow) list[wb + __popc(bal & ((1u << lane) - 1u))] = (int32_t)q;
}

// MINB: blocks per SM the register allocation is held to (3: 168 registers, 4:
// 128 with some spilled), a shape the tuner chooses; the arithmetic is the same
template <int MINB>
__global__ void __launch_bounds__(EST_THREADS, MINB) k_estimate_f32(GsProblem P, int level, const float *__restrict__ A,
                                                            const float *__restrict__ E, uint8_t *__restrict__ dec,
                                                            uint8_t *__restrict__ flag, unsigned long long *why_cnt,
                                                            float *__restrict__ dbg, const int32_t *__restrict__ list,
                                                            const unsigned *nlist)
{
    __shared__ float s_S[EST_SHARED * EST_THREADS];
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= (int64_t)*nlist) return;
    estimate_full_f32(P, level, A, E, (int64_t)list[t], dec, flag, why_cnt, dbg, s_S + threadIdx.x);
}

// cubes whose FP32 decision rests on one rank rule near its threshold
// (flag 0x80 | (rule + 1) << 3 | flipped rank) -> a compact list
__global__ void k_alt_list(const uint8_t *flag, int64_t n, int32_t *list, unsigned *nlist)
{
    int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    bool on = q < n && (flag[q] & 0x80);
    unsigned bal = __ballot_sync(0xffffffffu, on);
    if (!bal) return;
    unsigned lane = threadIdx.x & 31, base = 0;
    if (lane == 0) base = atomicAdd(nlist, (unsigned)__popc(bal));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (on) list[base + __popc(bal & ((1u << lane) - 1u))] = (int32_t)q;
}

// the listed cubes re-estimated under the flipped rank: the decision stands
// (flag 0) when it is the same with a margin outside the band and no other
// rule of the flipped estimate is near its threshold; otherwise FP64 decides
__global__ void __launch_bounds__(EST_THREADS) k_estimate_alt(GsProblem P, int level, const float *__restrict__ A,
                                                      const float *__restrict__ E, const int32_t *__restrict__ list,
                                                      const unsigned *nlist, const uint8_t *__restrict__ dec,
                                                      uint8_t *__restrict__ flag, unsigned long long *why_cnt)
{
    __shared__ float s_S[EST_SHARED * EST_THREADS];
    const int64_t nl = (int64_t)*nlist;
    for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < nl; t += (int64_t)gridDim.x * blockDim.x) {
    int64_t q = list[t];
    const unsigned code = flag[q];
    const int who = (int)((code >> 3) & 7u) - 1, altr = (int)(code & 7u);
    float tot = 0.f;
#pragma unroll
    for (int k = 0; k < 64; k++) tot += fabsf(A[q * 64 + k]);
    const float c = (float)P.c, prec = (float)P.precision;
    const float dA = MIXED_KAPPA * E[q] + 1e-7f * tot;
    float b2[6], rm2, sens2;
    estimate_bounds_sens(A + q * 64, s_S + threadIdx.x, b2, rm2, sens2, who < 0 ? altr : 0, who, who < 0 ? 0 : altr, nullptr);
    const float bAlt = 4.f * (dA + 1e-7f * tot) * (1.f + fminf(sens2, 1e4f));
    const float mc2 = fminf(fabsf(c - b2[0]), fabsf(b2[1] - c));
    const bool ok = rm2 > 32.f * dA + 1e-5f * tot && decide<float>(b2, c, prec, level, P.max_depth) == (int)dec[q] &&
                    mc2 > bAlt;
    flag[q] = ok ? 0 : 1;
    if (!ok && why_cnt) {
        atomicAdd(&why_cnt[0], 1ull);
        atomicAdd(&why_cnt[5], 1ull);
    }
    }
}

int gs_estimate_f32(const GsProblem &P, int level, const float *d_A, const float *d_err, int64_t n_cubes,
                    const uint64_t *d_parents, const uint8_t *d_vmask, uint8_t *d_dec, uint8_t *d_flag,
                    cudaStream_t st, unsigned long long *d_why, float *d_dbg)
{
    if (n_cubes <= 0) return GS_OK;
    int32_t *list = nullptr;
    unsigned *nlist = nullptr;
    int rc = gs_alloc((void **)&list, sizeof(int32_t) * (size_t)n_cubes, st);
    if (!rc) rc = gs_alloc((void **)&nlist, sizeof(unsigned), st);
    if (rc) { gs_free(list, st); return rc; }
    GS_CHECK(cudaMemsetAsync(nlist, 0, sizeof(unsigned), st));
    GS_LAUNCH(k_estimate_pre, (unsigned)((n_cubes + 255) / 256), 256, 0, st)(P, level, d_A, d_err, n_cubes, d_parents,
                                                                            d_vmask, d_dec, d_flag, d_why, d_dbg,
                                                                            list, nlist);
    const unsigned grid = (unsigned)((n_cubes + 127) / 128);
    rc = gs_tune_run("k_estimate_f32", n_cubes, 2, st, [&](int shape, unsigned long long *scratch) {
        unsigned long long *why = scratch ? (d_why ? scratch : nullptr) : d_why;
        if (shape == 0)
            GS_LAUNCH(k_estimate_f32<3>, grid, EST_THREADS, 0, st)(P, level, d_A, d_err, d_dec, d_flag, why, d_dbg, list, nlist);
        else
            GS_LAUNCH(k_estimate_f32<4>, grid, EST_THREADS, 0, st)(P, level, d_A, d_err, d_dec, d_flag, why, d_dbg, list, nlist);
    });
    gs_free(list, st);
    gs_free(nlist, st);
    if (rc) return rc;
    GS_CHECK(cudaGetLastError());
    return GS_OK;
}
__global__ void k_add_u64(unsigned long long *dst, const unsigned long long *v) { *dst += *v; }

// octets with a flagged child -> list of octet indices; counts flagged children
__global__ void k_octet_flags(const uint8_t *flag, int64_t n_oct, int64_t *cnt, unsigned long long *nflagged)
{
    int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= n_oct) return;
    uint64_t w = *(const uint64_t *)(flag + 8 * o);
    cnt[o] = w != 0;
    if (w && nflagged) {
        int k = 0;
        for (int c = 0; c < 8; c++) k += ((w >> (8 * c)) & 0xff) != 0;
        atomicAdd(nflagged, (unsigned long long)k);
    }
}
__global__ void k_octet_gather(const int64_t *off, int64_t n_oct, const uint64_t *parents, const uint8_t *flag,
                               uint64_t *sub_par, int64_t *sub_idx, uint8_t *sub_mask)
{
    int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= n_oct || off[o + 1] == off[o]) return;
    sub_par[off[o]] = parents[o];
    sub_idx[off[o]] = o;
    uint8_t m = 0;
    for (int c = 0; c < 8; c++)
        if (flag[8 * o + c]) m |= (uint8_t)(1u << c);
    sub_mask[off[o]] = m;
}
// flagged children of the re-evaluated octets -> a compact list (any order:
// each entry is estimated on its own), so the FP64 estimate runs full warps
__global__ void k_child_list(const uint8_t *sub_mask, int64_t n_sub, int32_t *list, unsigned *nlist)
{
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    bool on = t < n_sub * 8 && ((sub_mask[t >> 3] >> (t & 7)) & 1);
    unsigned bal = __ballot_sync(0xffffffffu, on);
    if (!bal) return;
    unsigned lane = threadIdx.x & 31, base = 0;
    if (lane == 0) base = atomicAdd(nlist, (unsigned)__popc(bal));
    base = __shfl_sync(0xffffffffu, base, 0);
    if (on) list[base + __popc(bal & ((1u << lane) - 1u))] = (int32_t)t;
}
// the FP64 decisions replace the flagged children's FP32 ones
__global__ void k_octet_scatter(const uint8_t *sub_dec, const int64_t *sub_idx, const uint8_t *sub_mask, int64_t n_sub,
                                uint8_t *dec)
{
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= n_sub * 8) return;
    if (!((sub_mask[t >> 3] >> (t & 7)) & 1)) return;
    dec[sub_idx[t >> 3] * 8 + (t & 7)] = sub_dec[t];
}
// debug: largest change of L or U between the FP32 and FP64 estimates,
// relative to (dA + 1e-7 sum|A|)(1 + s), over cubes whose rank rules are not
// within their band (those get the rank-flip allowance instead)
__global__ void k_band_ratio(const float *dbg, const double *b64, const uint8_t *d64, int64_t n, unsigned *maxbits)
{
    int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n || d64[q] == DEC_INVALID) return;
    const float *o = dbg + 6 * q;
    if (o[4] <= 0.f || o[5] != 0.f) return;
    double dl = fabs((double)o[0] - b64[6 * q]), du = fabs((double)o[1] - b64[6 * q + 1]);
    double den = ((double)o[3] + 1e-7 * (double)o[4]) * (1.0 + (double)o[2]);
    float r = (float)(fmax(dl, du) / den);
    atomicMax(maxbits, __float_as_uint(r));
}

// debug: largest |A32 - A64| / E over a chunk, as float bits (non-negative)
__global__ void k_err_ratio(const float *A32, const float *E, const double *A64, int64_t n, unsigned *maxbits)
{
    int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    double mx = 0;
    for (int t = 0; t < 64; t++) mx = fmax(mx, fabs((double)A32[q * 64 + t] - A64[q * 64 + t]));
    float e = E[q];
    if (e > 0.f) {
        float r = (float)(mx / e);
        atomicMax(maxbits, __float_as_uint(r));
    }
}

__global__ void k_count_mismatch(const uint8_t *a, const uint8_t *b, int64_t n, unsigned long long *mism)
{
    int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (q >= n) return;
    // cube sets depend on discard / keep and split / accept; accepted vs forced is bookkeeping
    unsigned x = a[q], y = b[q];
    if (x == DEC_FORCED) x = DEC_ACCEPT;
    if (y == DEC_FORCED) y = DEC_ACCEPT;
    if (x != y) atomicAdd(mism, 1ull);
}

// one chunk of a level in mixed precision; dec receives the final decisions
// d_why: [0..2] flag reasons (bounds band, precision band, zero tensor), [3] low 32 bits = float bits of
// the largest |A32 - A64| / E seen in debug mode, [4] the same for the band ratio, [5] flags through a rank
// rule, [10] cubes decided without the SVD (corner values straddle c, range
// and distance from rank one exclude it, or no atom reaches them)
__global__ void k_gather_mol(const int64_t *__restrict__ si, int64_t m, const int32_t *__restrict__ mol,
                             int32_t *__restrict__ sub_mol)
{
    int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (t < m) sub_mol[t] = mol[si[t]];
}

int gs_level_mixed(const GsProblem &P, int level, const uint64_t *d_parents, int64_t n_oct, uint8_t *d_dec,
                   unsigned long long *d_pairs, unsigned long long *d_rechecked, unsigned long long *d_mism,
                   bool both, cudaStream_t st, cudaEvent_t *ev, unsigned long long *d_why,
                   const GsProblem *d_probs, const int32_t *d_mol, const uint8_t *d_vmask)
{
    float *A = nullptr, *E = nullptr;
    uint8_t *flag = nullptr;
    int rc = gs_alloc((void **)&A, sizeof(float) * 64 * 8 * (size_t)n_oct, st);
    if (!rc) rc = gs_alloc((void **)&E, sizeof(float) * 8 * (size_t)n_oct, st);
    if (!rc) rc = gs_alloc((void **)&flag, 8 * (size_t)n_oct, st);
    float *dbg = nullptr;
    if (!rc && both) rc = gs_alloc((void **)&dbg, sizeof(float) * 6 * 8 * (size_t)n_oct, st);
    // the counter block holds the atom-octet count 16 slots after the pair count
    if (!rc)
        rc = gs_accum_f32(P, level, d_parents, d_vmask, n_oct, A, E, d_pairs, st, ev, d_pairs + 16, d_probs,
                          d_mol);
    if (!rc) rc = gs_estimate_f32(P, level, A, E, n_oct * 8, d_parents, d_vmask, d_dec, flag, st, d_why, dbg);
    if (!rc) {
        // decisions resting on one rank rule near its threshold
        int32_t *lst = nullptr;
        unsigned *nl = nullptr;
        rc = gs_alloc((void **)&lst, sizeof(int32_t) * 8 * (size_t)n_oct, st);
        if (!rc) rc = gs_alloc((void **)&nl, sizeof(unsigned), st);
        if (!rc) {
            unsigned nb = (unsigned)((n_oct * 8 + 127) / 128);
            cudaMemsetAsync(nl, 0, sizeof(unsigned), st);
            GS_LAUNCH(k_alt_list, nb, 128, 0, st)(flag, n_oct * 8, lst, nl);
            GS_LAUNCH(k_estimate_alt, 152 * 4, 128, 0, st)(P, level, A, E, lst, nl, d_dec, flag, d_why);
        }
        gs_free(lst, st); gs_free(nl, st);
    }
    // flagged octets -> FP64
    int64_t *cnt = nullptr, *tot = nullptr;
    if (!rc) rc = gs_alloc((void **)&cnt, sizeof(int64_t) * (size_t)(n_oct + 1), st);
    if (!rc) rc = gs_alloc((void **)&tot, sizeof(int64_t), st);
    if (!rc) {
        cudaMemsetAsync(cnt + n_oct, 0, sizeof(int64_t), st);
        GS_LAUNCH(k_octet_flags, (unsigned)((n_oct + 255) / 256), 256, 0, st)(flag, n_oct, cnt, d_rechecked);
        rc = gs_scan_i64(cnt, n_oct + 1, tot, st);
    }
    int64_t nsub = 0;
    if (!rc) {
        cudaError_t e = cudaMemcpyAsync(&nsub, tot, sizeof(int64_t), cudaMemcpyDeviceToHost, st);
        if (e == cudaSuccess) e = gs_sync(st);
        if (e != cudaSuccess) rc = gs_fail_cuda(e, "recheck count", __FILE__, __LINE__);
    }
    if (!rc && nsub > 0) {
        uint64_t *sp = nullptr;
        int64_t *si = nullptr;
        double *A64 = nullptr;
        uint8_t *sd = nullptr, *sm = nullptr;
        rc = gs_alloc((void **)&sp, sizeof(uint64_t) * (size_t)nsub, st);
        if (!rc) rc = gs_alloc((void **)&si, sizeof(int64_t) * (size_t)nsub, st);
        if (!rc) rc = gs_alloc((void **)&sm, (size_t)nsub, st);
        if (!rc) rc = gs_alloc((void **)&A64, sizeof(double) * 64 * 8 * (size_t)nsub, st);
        if (!rc) rc = gs_alloc((void **)&sd, 8 * (size_t)nsub, st);
        int32_t *smol = nullptr;
        if (!rc && d_mol) rc = gs_alloc((void **)&smol, sizeof(int32_t) * (size_t)nsub, st);
        if (!rc) {
            GS_LAUNCH(k_octet_gather, (unsigned)((n_oct + 255) / 256), 256, 0, st)(cnt, n_oct, d_parents, flag, sp, si,
                                                                                  sm);
            if (d_mol) GS_LAUNCH(k_gather_mol, (unsigned)((nsub + 255) / 256), 256, 0, st)(si, nsub, d_mol, smol);
            // only the flagged children are accumulated and estimated in FP64
            rc = gs_accum_f64(P, level, sp, sm, nsub, A64, nullptr, st, nullptr, d_probs, smol);
        }
        int32_t *lst = nullptr;
        unsigned *nl = nullptr;
        if (!rc) rc = gs_alloc((void **)&lst, sizeof(int32_t) * 8 * (size_t)nsub, st);
        if (!rc) rc = gs_alloc((void **)&nl, sizeof(unsigned), st);
        if (!rc) {
            unsigned nb = (unsigned)((nsub * 8 + 127) / 128);
            cudaMemsetAsync(nl, 0, sizeof(unsigned), st);
            GS_LAUNCH(k_child_list, nb, 128, 0, st)(sm, nsub, lst, nl);
            launch_estimate_f64(P, level, A64, nsub * 8, sp, sm, sd, nullptr, lst, nl, st);
        }
        gs_free(lst, st); gs_free(nl, st);
        if (!rc) GS_LAUNCH(k_octet_scatter, (unsigned)((nsub * 8 + 255) / 256), 256, 0, st)(sd, si, sm, nsub, d_dec);
        gs_free(sp, st); gs_free(si, st); gs_free(sm, st); gs_free(A64, st); gs_free(sd, st); gs_free(smol, st);
    }
    gs_free(cnt, st); gs_free(tot, st);
    if (!rc && both) {
        // debug: FP64 on every octet; count final decisions that disagree and
        // record the largest |A32 - A64| / E
        double *A64 = nullptr, *b64 = nullptr;
        uint8_t *d64 = nullptr;
        rc = gs_alloc((void **)&A64, sizeof(double) * 64 * 8 * (size_t)n_oct, st);
        if (!rc) rc = gs_alloc((void **)&b64, sizeof(double) * 6 * 8 * (size_t)n_oct, st);
        if (!rc) rc = gs_alloc((void **)&d64, 8 * (size_t)n_oct, st);
        if (!rc)
            rc = gs_accum_f64(P, level, d_parents, d_vmask, n_oct, A64, nullptr, st, nullptr, d_probs, d_mol);
        if (!rc) rc = gs_estimate_f64(P, level, A64, n_oct * 8, d_parents, d_vmask, d64, b64, st);
        if (!rc) {
            unsigned nb = (unsigned)((n_oct * 8 + 255) / 256);
            GS_LAUNCH(k_count_mismatch, nb, 256, 0, st)(d_dec, d64, n_oct * 8, d_mism);
            GS_LAUNCH(k_err_ratio, nb, 256, 0, st)(A, E, A64, n_oct * 8, (unsigned *)(d_why + 3));
            GS_LAUNCH(k_band_ratio, nb, 256, 0, st)(dbg, b64, d64, n_oct * 8, (unsigned *)(d_why + 4));
        }
        gs_free(A64, st); gs_free(b64, st); gs_free(d64, st);
    }
    gs_free(A, st);
    gs_free(E, st);
    gs_free(dbg, st);
    gs_free(flag, st);
    if (rc) return rc;
    GS_CHECK(cudaGetLastError());
    return GS_OK;
}

// ================================================================ batched form
// Several molecules share one level loop: the octets of all molecules sit in
// one array, molecule by molecule, with the molecule's index (its row in a
// device table of problem records) beside each octet.  Compaction is stable,
// so every level's arrays stay grouped by molecule and each molecule's
// octets keep the order a single-molecule run gives them.

// root blocks of every molecule: keys in the molecule's own lattice, the
// valid children (inside the molecule's root grid) and the molecule index.
// tab[g] = {first octet, bx, by, nroot x, nroot y, nroot z}; base[G] = total
__global__ void k_root_blocks_batch(const int64_t *__restrict__ tab, int G, int64_t n, uint64_t *__restrict__ keys,
                                    uint8_t *__restrict__ vmask, int32_t *__restrict__ mol)
{
    const int64_t o = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (o >= n) return;
    int lo = 0, hi = G - 1;   // last g with tab[g].first <= o
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (tab[6 * mid] <= o) lo = mid;
        else hi = mid - 1;
    }
    const int64_t *t = tab + 6 * lo;
    const int64_t r = o - t[0], bx = t[1], by = t[2];
    const int64_t I = r % bx, J = (r / bx) % by, K = r / (bx * by);
    uint8_t m = 0;
    for (int c = 0; c < 8; c++) {
        const int64_t x = 2 * I + (c & 1), y = 2 * J + ((c >> 1) & 1), z = 2 * K + (c >> 2);
        if (x < t[3] && y < t[4] && z < t[5]) m |= (uint8_t)(1u << c);
    }
    keys[o] = gk_make(I, J, K, GT_CUBE, 0);
    vmask[o] = m;
    mol[o] = lo;
}

int gs_root_blocks_batch(const GsProblem *probs, int G, uint64_t **d_keys, uint8_t **d_vmask, int32_t **d_mol,
                         int64_t *n, cudaStream_t st)
{
    *d_keys = nullptr; *d_vmask = nullptr; *d_mol = nullptr; *n = 0;
    std::vector<int64_t> tab(6 * (size_t)G);
    int64_t total = 0;
    for (int g = 0; g < G; g++) {
        const int64_t bx = (probs[g].nroot[0] + 1) / 2, by = (probs[g].nroot[1] + 1) / 2,
                      bz = (probs[g].nroot[2] + 1) / 2;
        int64_t *t = &tab[6 * (size_t)g];
        t[0] = total; t[1] = bx; t[2] = by;
        t[3] = probs[g].nroot[0]; t[4] = probs[g].nroot[1]; t[5] = probs[g].nroot[2];
        total += bx * by * bz;
    }
    int64_t *d_tab = nullptr;
    int rc = gs_alloc((void **)&d_tab, sizeof(int64_t) * tab.size(), st);
    if (!rc) rc = gs_alloc((void **)d_keys, sizeof(uint64_t) * (size_t)total, st);
    if (!rc) rc = gs_alloc((void **)d_vmask, (size_t)total, st);
    if (!rc) rc = gs_alloc((void **)d_mol, sizeof(int32_t) * (size_t)total, st);
    if (!rc) {
        cudaError_t e = cudaMemcpyAsync(d_tab, tab.data(), sizeof(int64_t) * tab.size(), cudaMemcpyHostToDevice, st);
        if (e != cudaSuccess) rc = gs_fail_cuda(e, "root table", __FILE__, __LINE__);
    }
    if (!rc) GS_LAUNCH(k_root_blocks_batch, (unsigned)((total + 255) / 256), 256, 0, st)(d_tab, G, total, *d_keys,
                                                                                     *d_vmask, *d_mol);
    gs_free(d_tab, st);
    if (rc) {
        gs_free(*d_keys, st); gs_free(*d_vmask, st); gs_free(*d_mol, st);
        *d_keys = nullptr; *d_vmask = nullptr; *d_mol = nullptr;
        return rc;
    }
    GS_CHECK(cudaGetLastError());
    *n = total;
    return GS_OK;
}

// per-molecule decision counts: cnt[g * 5 + k] (examined, discarded,
// accepted, forced, split).  The cubes are grouped by molecule, so the lanes
// of a warp mostly share one (molecule, decision) pair and one atomic per
// pair and warp suffices.
__global__ void __launch_bounds__(256) k_level_count_mol(const uint8_t *__restrict__ dec, int64_t n,
                                                         const int32_t *__restrict__ mol,
                                                         unsigned long long *__restrict__ cnt)
{
    const int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    const unsigned full = 0xffffffffu;
    unsigned d = q < n ? dec[q] : DEC_INVALID;
    const int g = q < n ? mol[q >> 3] : 0;
    // slot 0 (examined) for every valid cube, then the decision's own slot
    const int k = d == DEC_DISCARD ? 1 : d == DEC_ACCEPT ? 2 : d == DEC_FORCED ? 3 : d == DEC_SPLIT ? 4 : -1;
    const unsigned key0 = d != DEC_INVALID ? (unsigned)g * 8u : 0xFFFFFFFFu;
    const unsigned p0 = __match_any_sync(full, key0);
    if (key0 != 0xFFFFFFFFu && (threadIdx.x & 31) == __ffs(p0) - 1)
        atomicAdd(&cnt[(int64_t)g * 5], (unsigned long long)__popc(p0));
    const unsigned key1 = k >= 0 ? (unsigned)g * 8u + (unsigned)k : 0xFFFFFFFFu;
    const unsigned p1 = __match_any_sync(full, key1);
    if (key1 != 0xFFFFFFFFu && (threadIdx.x & 31) == __ffs(p1) - 1)
        atomicAdd(&cnt[(int64_t)g * 5 + k], (unsigned long long)__popc(p1));
}

int gs_level_count_mol(const uint8_t *d_dec, int64_t n_cubes, const int32_t *d_mol, unsigned long long *d_cnt,
                       cudaStream_t st)
{
    if (n_cubes <= 0) return GS_OK;
    GS_LAUNCH(k_level_count_mol, (unsigned)((n_cubes + 255) / 256), 256, 0, st)(d_dec, n_cubes, d_mol, d_cnt);
    GS_CHECK(cudaGetLastError());
    return GS_OK;
}

// accepted cubes of one compaction part to their molecules' arrays: cube j
// of the part (molecule g) goes to outs[g][j + q0 + shift[g]], q0 being the
// part's first slot among its level's accepted cubes and shift[g] the
// molecule's count over the earlier levels minus its first slot in this one
// (cap[g]: the size of molecule g's array; a slot outside it, which only
// cubes out of molecule order could give, sets GS_ST_CAPACITY instead)
__global__ void k_scatter_cubes(const uint64_t *__restrict__ acc, const int32_t *__restrict__ acc_mol, int64_t n,
                                int64_t q0, const int64_t *__restrict__ shift, uint64_t *const *__restrict__ outs,
                                const int64_t *__restrict__ cap, unsigned *status)
{
    const int64_t j = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= n) return;
    const int g = acc_mol[j];
    const int64_t d = j + q0 + shift[g];
    if (d < 0 || d >= cap[g]) {
        atomicOr(status, GS_ST_CAPACITY);
        return;
    }
    outs[g][d] = acc[j];
}

int gs_scatter_cubes(const uint64_t *d_acc, const int32_t *d_acc_mol, int64_t n, int64_t q0, const int64_t *d_shift,
                     uint64_t *const *d_outs, const int64_t *d_cap, unsigned *d_status, cudaStream_t st)
{
    if (n <= 0) return GS_OK;
    GS_LAUNCH(k_scatter_cubes, (unsigned)((n + 255) / 256), 256, 0, st)(d_acc, d_acc_mol, n, q0, d_shift, d_outs,
                                                                        d_cap, d_status);
    GS_CHECK(cudaGetLastError());
    return GS_OK;
}
