// Region evaluation (the hot loop): for each region on the eval list, the
// nested Clenshaw-Curtis pair Q_N (coarse, N intervals per dimension) and Q_2N
// (fine, 2N intervals) of the bubble integrand, and err = |Q_N - Q_2N|
// (Sec. 3; Listing 3 evaluates the four children of a split this way).
//
// Integrand (Sec. 2, Eq. chi_ph / chi_pp after the Matsubara sum):
//   ph: f_l(k) f_m(k+q) F(e(k), e(k+q)),   pp: f_l(k) f_m(q-k) F(e(k), -e(q-k))
//   F(e1, e2) = [tanh(e1/2T) - tanh(e2/2T)] / (2 (e1 - e2))
// which equals [nF(e2) - nF(e1)]/(e1 - e2) for ph and, with e2 -> -e(q-k),
// [1 - nF(e1) - nF(e(q-k))]/(e1 + e(q-k)) for pp.  F is evaluated without
// cancellation from v = exp(-|x|), x = e/2T:
//   |d| <= 1/16, d = (e1 - e2)/2T:  F = (1/4T) sinhc(d) sech x1 sech x2
//                                      (tanh a - tanh b = sinh(a-b) sech a sech b)
//   same sign:      F = s (u2 - u1) / ((1+u1)(1+u2)(e1 - e2)),  u = v^2
//   opposite sign:  F = s (1 - u1 u2) / ((1+u1)(1+u2)(e1 - e2))
// with sech x = 2v/(1+u) and s the sign of x1.  One exp per energy and one
// division per node.
//
// Data reuse inside a region (tensor-product hoisting): the 2N+1 node
// abscissae per dimension are cos/sin rotations of the region centre, taken
// from sincospi of the exact dyadic centre and a per-level table of the node
// offsets, so a region costs 2 sincospi instead of 2(2N+1)^2 cos/sin.  The
// dispersion is affine in cos ky for fixed kx, e = A(kx) + B(kx) cos ky, and
// each form factor is X(kx)^T C Y(ky) with X = (1, cos kx, sin kx).
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <type_traits>

#include "paid_internal.cuh"

namespace paid {

// rule variant v = (N - 4) / 2: N = 4 (5 x 5 coarse inside 9 x 9 fine), 6 (7 inside
// 13), and for the shared-partition kernel only 8, 10, 12 (13 inside 25)
__constant__ double c_wf[kRuleVariants][2 * kMaxRuleN + 1];   // fine CC weights on [-1, 1]
__constant__ double c_wc[kRuleVariants][kMaxRuleN + 1];       // coarse CC weights
__constant__ double c_t[kRuleVariants][2 * kMaxRuleN + 1];    // fine nodes t_i = cos(i pi / 2N)
__constant__ double c_co[kRuleVariants][kMaxLevel + 1][kMaxRuleN + 1];  // cos(pi 2^-L t_i), i <= N
__constant__ double c_so[kRuleVariants][kMaxLevel + 1][kMaxRuleN + 1];  // sin(pi 2^-L t_i)
__constant__ double c_ff[9][3][3];                // f_n = sum_ab C[a][b] X_a Y_b
__constant__ float c_wf32[2][2 * kMaxRuleNLow + 1];  // FP32 copies for the FP32 path
__constant__ float2 c_wfdf[2][2 * kMaxRuleNLow + 1]; // (hi, lo) pairs for the float-float path
__constant__ float2 c_wcdf[2][kMaxRuleNLow + 1];
__constant__ float2 c_exp2tab[64];                // 2^(j/64) as (hi, lo), j = 0..63
__constant__ float2 c_codf[2][kMaxLevel + 1][kMaxRuleNLow + 1];  // c_co / c_so as (hi, lo)
__constant__ float2 c_sodf[2][kMaxLevel + 1][kMaxRuleNLow + 1];
__constant__ float2 c_ffdf[9][3][3];              // c_ff as (hi, lo)
__constant__ float c_wc32[2][kMaxRuleNLow + 1];
__constant__ float c_ff32[9][3][3];
// the non-zero terms of c_ff: f_n = sum_{k < c_ffn[n]} c_ffc[n][k] X_a Y_b, a = c_ffa, b = c_ffb
__constant__ int c_ffn[9];
__constant__ int c_ffa[9][2];
__constant__ int c_ffb[9][2];
__constant__ double c_ffc[9][2];
__constant__ double c_exp2d[64];                  // 2^(j/64), j = 0..63 (FP64 exp of the group path)
// The FP32-pipe group kernel's tables, in global memory (lanes read different
// entries, which constant memory would serialise): c_co and c_so as
// float-float (cos hi, cos lo, sin hi, sin lo), and per pair (l, m) the
// non-zero terms of f_l f_m' in order, the coefficient c_ffc[l] c_ffc[m] as
// float-float and the index 9 ac + bd of its product moment as the third
// word's bits (-1 ends the list)
__device__ float4 g_cosine[kRuleVariants][kMaxLevel + 1][kMaxRuleN + 1];
__device__ float4 g_terms[9][9][4];

// Clenshaw-Curtis weights for n intervals (n even), from the cosine-series
// form of the rule: w_j = (c_j / n) (1 - sum_{k=1}^{n/2} b_k cos(2 k j pi/n)/(4k^2 - 1)).
static void cc_weights(int n, double* w)
{
    for (int j = 0; j <= n; ++j) {
        double acc = 1.0;
        for (int k = 1; k <= n / 2; ++k) {
            double bk = (2 * k == n) ? 1.0 : 2.0;
            acc -= bk * std::cos(2.0 * k * j * kPi / n) / (4.0 * k * k - 1.0);
        }
        w[j] = ((j == 0 || j == n) ? 1.0 : 2.0) / n * acc;
    }
}

static cudaError_t group_kernel_attributes();

cudaError_t init_rule_tables(int device)
{
    // contexts may be created by several threads at once: one of them fills the
    // device's tables, the others wait for it
    static std::mutex mutex;
    static bool done[64] = {false};
    if (device < 0 || device >= 64) return cudaErrorInvalidDevice;
    const std::lock_guard<std::mutex> lock(mutex);
    if (done[device]) return cudaSuccess;
    double wf[kRuleVariants][2 * kMaxRuleN + 1] = {}, wc[kRuleVariants][kMaxRuleN + 1] = {};
    double t[kRuleVariants][2 * kMaxRuleN + 1] = {};
    double co[kRuleVariants][kMaxLevel + 1][kMaxRuleN + 1] = {};
    double so[kRuleVariants][kMaxLevel + 1][kMaxRuleN + 1] = {};
    const int Ns[kRuleVariants] = {4, 6, 8, 10, 12};
    for (int v = 0; v < kRuleVariants; ++v) {
        int N = Ns[v];
        cc_weights(2 * N, wf[v]);
        cc_weights(N, wc[v]);
        for (int i = 0; i <= 2 * N; ++i) t[v][i] = std::cos(i * kPi / (2 * N));
        t[v][N] = 0.0;
        for (int L = 0; L <= kMaxLevel; ++L)
            for (int i = 0; i <= N; ++i) {
                double o = std::ldexp(kPi, -L) * t[v][i];   // half side pi 2^-L times t_i
                co[v][L][i] = std::cos(o);
                so[v][L][i] = std::sin(o);
            }
    }
    const double r2 = std::sqrt(2.0);
    double ff[9][3][3] = {};
    ff[0][0][0] = 1.0;                      // 1
    ff[1][1][0] = 1.0; ff[1][0][1] = 1.0;   // cx + cy
    ff[2][1][0] = 1.0; ff[2][0][1] = -1.0;  // cx - cy
    ff[3][2][0] = r2;                       // sqrt2 sx
    ff[4][0][2] = r2;                       // sqrt2 sy
    ff[5][1][1] = 2.0;                      // 2 cx cy
    ff[6][2][2] = 2.0;                      // 2 sx sy
    ff[7][2][1] = 2.0;                      // 2 sx cy
    ff[8][1][2] = 2.0;                      // 2 cx sy
    float wf32[2][2 * kMaxRuleNLow + 1], wc32[2][kMaxRuleNLow + 1], ff32[9][3][3];
    for (int v = 0; v < 2; ++v) {
        for (int i = 0; i < 2 * kMaxRuleNLow + 1; ++i) wf32[v][i] = float(wf[v][i]);
        for (int i = 0; i < kMaxRuleNLow + 1; ++i) wc32[v][i] = float(wc[v][i]);
    }
    for (int a = 0; a < 9; ++a)
        for (int b = 0; b < 3; ++b)
            for (int c = 0; c < 3; ++c) ff32[a][b][c] = float(ff[a][b][c]);
    float2 wfdf[2][2 * kMaxRuleNLow + 1], wcdf[2][kMaxRuleNLow + 1], e2t[64];
    auto split = [](double x) { float hi = float(x); return make_float2(hi, float(x - double(hi))); };
    for (int v = 0; v < 2; ++v) {
        for (int i = 0; i < 2 * kMaxRuleNLow + 1; ++i) wfdf[v][i] = split(wf[v][i]);
        for (int i = 0; i < kMaxRuleNLow + 1; ++i) wcdf[v][i] = split(wc[v][i]);
    }
    for (int j = 0; j < 64; ++j) e2t[j] = split(std::exp2(j / 64.0));
    float2 codf[2][kMaxLevel + 1][kMaxRuleNLow + 1], sodf[2][kMaxLevel + 1][kMaxRuleNLow + 1];
    float2 ffdf[9][3][3];
    for (int v = 0; v < 2; ++v)
        for (int L = 0; L <= kMaxLevel; ++L)
            for (int i = 0; i <= kMaxRuleNLow; ++i) {
                codf[v][L][i] = split(co[v][L][i]);
                sodf[v][L][i] = split(so[v][L][i]);
            }
    for (int a = 0; a < 9; ++a)
        for (int b = 0; b < 3; ++b)
            for (int c = 0; c < 3; ++c) ffdf[a][b][c] = split(ff[a][b][c]);
    cudaError_t e;
    if ((e = cudaMemcpyToSymbol(c_codf, codf, sizeof(codf))) != cudaSuccess) return e;
    if ((e = cudaMemcpyToSymbol(c_sodf, sodf, sizeof(sodf))) != cudaSuccess) return e;
    if ((e = cudaMemcpyToSymbol(c_ffdf, ffdf, sizeof(ffdf))) != cudaSuccess) return e;
    if ((e = cudaMemcpyToSymbol(c_wfdf, wfdf, sizeof(wfdf))) != cudaSuccess) return e;
    if ((e = cudaMemcpyToSymbol(c_wcdf, wcdf, sizeof(wcdf))) != cudaSuccess) return e;
    if ((e = cudaMemcpyToSymbol(c_exp2tab, e2t, sizeof(e2t))) != cudaSuccess) return e;
    if ((e = cudaMemcpyToSymbol(c_wf32, wf32, sizeof(wf32))) != cudaSuccess) return e;
    if ((e = cudaMemcpyToSymbol(c_wc32, wc32, sizeof(wc32))) != cudaSuccess) return e;
    if ((e = cudaMemcpyToSymbol(c_ff32, ff32, sizeof(ff32))) != cudaSuccess) return e;
    if ((e = cudaMemcpyToSymbol(c_wf, wf, sizeof(wf))) != cudaSuccess) return e;
    if ((e = cudaMemcpyToSymbol(c_wc, wc, sizeof(wc))) != cudaSuccess) return e;
    if ((e = cudaMemcpyToSymbol(c_t, t, sizeof(t))) != cudaSuccess) return e;
    if ((e = cudaMemcpyToSymbol(c_co, co, sizeof(co))) != cudaSuccess) return e;
    if ((e = cudaMemcpyToSymbol(c_so, so, sizeof(so))) != cudaSuccess) return e;
    if ((e = cudaMemcpyToSymbol(c_ff, ff, sizeof(ff))) != cudaSuccess) return e;
    int ffn[9] = {}, ffa[9][2] = {}, ffb[9][2] = {};
    double ffc[9][2] = {};
    for (int n = 0; n < 9; ++n)
        for (int a = 0; a < 3; ++a)
            for (int b = 0; b < 3; ++b)
                if (ff[n][a][b] != 0.0) {
                    ffa[n][ffn[n]] = a;
                    ffb[n][ffn[n]] = b;
                    ffc[n][ffn[n]] = ff[n][a][b];
                    ++ffn[n];
                }
    if ((e = cudaMemcpyToSymbol(c_ffn, ffn, sizeof(ffn))) != cudaSuccess) return e;
    if ((e = cudaMemcpyToSymbol(c_ffa, ffa, sizeof(ffa))) != cudaSuccess) return e;
    if ((e = cudaMemcpyToSymbol(c_ffb, ffb, sizeof(ffb))) != cudaSuccess) return e;
    if ((e = cudaMemcpyToSymbol(c_ffc, ffc, sizeof(ffc))) != cudaSuccess) return e;
    float4 cosine[kRuleVariants][kMaxLevel + 1][kMaxRuleN + 1];   // 31 KB
    for (int v = 0; v < kRuleVariants; ++v)
        for (int L = 0; L <= kMaxLevel; ++L)
            for (int i = 0; i <= kMaxRuleN; ++i) {
                const float2 c = split(co[v][L][i]), sn = split(so[v][L][i]);
                cosine[v][L][i] = make_float4(c.x, c.y, sn.x, sn.y);
            }
    if ((e = cudaMemcpyToSymbol(g_cosine, cosine, sizeof(cosine))) != cudaSuccess) return e;
    float4 terms[9][9][4];
    auto bits = [](int i) { float f; std::memcpy(&f, &i, sizeof(f)); return f; };
    for (int l = 0; l < 9; ++l)
        for (int m = 0; m < 9; ++m) {
            int k = 0;
            for (int k1 = 0; k1 < ffn[l]; ++k1)
                for (int k2 = 0; k2 < ffn[m]; ++k2) {
                    const float2 c = split(ffc[l][k1] * ffc[m][k2]);
                    const int ac = 3 * ffa[l][k1] + ffa[m][k2], bd = 3 * ffb[l][k1] + ffb[m][k2];
                    terms[l][m][k++] = make_float4(c.x, c.y, bits(9 * ac + bd), 0.0f);
                }
            for (; k < 4; ++k) terms[l][m][k] = make_float4(0.0f, 0.0f, bits(-1), 0.0f);
        }
    if ((e = cudaMemcpyToSymbol(g_terms, terms, sizeof(terms))) != cudaSuccess) return e;
    double e2d[64];
    for (int j = 0; j < 64; ++j) e2d[j] = std::exp2(j / 64.0);
    if ((e = cudaMemcpyToSymbol(c_exp2d, e2d, sizeof(e2d))) != cudaSuccess) return e;
    if ((e = group_kernel_attributes()) != cudaSuccess) return e;
    done[device] = true;
    return cudaSuccess;
}

// ---------------------------------------------------------------------------
// FP64 bubble kernel F(e1, e2) (see the file header), inv2T = 1/2T, inv4T = 1/4T.
__device__ __forceinline__ double bubble_F(double e1, double e2, double inv2T, double inv4T)
{
    const double diff = e1 - e2;
    const double d = diff * inv2T;
    const double x1 = e1 * inv2T, x2 = e2 * inv2T;
    const double v1 = exp(-fabs(x1)), v2 = exp(-fabs(x2));
    const double u1 = v1 * v1, u2 = v2 * v2;
    const double p = (1.0 + u1) * (1.0 + u2);
    const bool near = fabs(d) <= 0.0625;
    const bool neg1 = x1 < 0.0;
    const bool same = neg1 == (x2 < 0.0);
    double far = same ? (u2 - u1) : fma(-u1, u2, 1.0);
    far = neg1 ? -far : far;
    const double d2 = d * d;
    const double sinhc = fma(d2, fma(d2, fma(d2, fma(d2, 1.0 / 362880.0, 1.0 / 5040.0),
                                              1.0 / 120.0), 1.0 / 6.0), 1.0);
    const double nearv = (4.0 * inv4T) * (v1 * v2) * sinhc;
    const double num = near ? nearv : far;
    const double den = near ? p : p * diff;
    return num / den;
}

// Sum of the fine (w2) and coarse (w1) tensor rules over one region of a
// trigonometric-path kind (PH, PP, OVERLAP), in FP64.  SHARED: the kernel F at node
// (i, j) is read from fp[32 (i NF + j)].
template <int N, int KIND, bool SHARED = false>
__device__ __forceinline__ void region_trig_fp64(int v, uint32_t L, uint32_t ix, uint32_t iy,
                                                 QTrig tq, int l, int m, const DevBatch& B,
                                                 Lattice lat, double& s2, double& s1,
                                                 const double* fp = nullptr)
{
    constexpr int NF = 2 * N + 1;
    const double inv2T = B.inv2T, inv4T = B.inv4T;
    // exact dyadic centre / pi: -1 + (2 ix + 1) 2^-L
    double sxc, cxc, syc, cyc;
    sincospi(fma(double(2 * ix + 1), ldexp(1.0, -int(L)), -1.0), &sxc, &cxc);
    sincospi(fma(double(2 * iy + 1), ldexp(1.0, -int(L)), -1.0), &syc, &cyc);

    double cy[NF], sy[NF], cy2[NF], sy2[NF];
#pragma unroll
    for (int j = 0; j < NF; ++j) {
        const int jj = j <= N ? j : 2 * N - j;
        const double co = c_co[v][L][jj];
        const double so = j <= N ? c_so[v][L][jj] : -c_so[v][L][jj];
        cy[j] = fma(cyc, co, -syc * so);
        sy[j] = fma(syc, co, cyc * so);
        if (KIND == PP) {   // q - k
            cy2[j] = fma(tq.cqy, cy[j], tq.sqy * sy[j]);
            sy2[j] = fma(tq.sqy, cy[j], -tq.cqy * sy[j]);
        } else {            // k + q
            cy2[j] = fma(cy[j], tq.cqy, -sy[j] * tq.sqy);
            sy2[j] = fma(sy[j], tq.cqy, cy[j] * tq.sqy);
        }
    }
    double Cl[3][3], Cm[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) { Cl[a][b] = c_ff[l][a][b]; Cm[a][b] = c_ff[m][a][b]; }

    const double tA = -2.0 * lat.t, tB = -4.0 * lat.tp;
    double fine = 0.0, coarse = 0.0;
#pragma unroll 1
    for (int i = 0; i < NF; ++i) {
        const int ii = i <= N ? i : 2 * N - i;
        const double co = c_co[v][L][ii];
        const double so = i <= N ? c_so[v][L][ii] : -c_so[v][L][ii];
        const double cx = fma(cxc, co, -sxc * so);
        const double sx = fma(sxc, co, cxc * so);
        double cx2, sx2;
        if (KIND == PP) { cx2 = fma(tq.cqx, cx, tq.sqx * sx); sx2 = fma(tq.sqx, cx, -tq.cqx * sx); }
        else            { cx2 = fma(cx, tq.cqx, -sx * tq.sqx); sx2 = fma(sx, tq.cqx, cx * tq.sqx); }
        // e = A + B cos ky along this row
        const double A1 = fma(tA, cx, -lat.mu), B1 = fma(tB, cx, tA);
        const double A2 = fma(tA, cx2, -lat.mu), B2 = fma(tB, cx2, tA);
        double ul[3], um[3];
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            ul[b] = fma(Cl[2][b], sx, fma(Cl[1][b], cx, Cl[0][b]));
            um[b] = fma(Cm[2][b], sx2, fma(Cm[1][b], cx2, Cm[0][b]));
        }
        double rf = 0.0, rc = 0.0;
#pragma unroll
        for (int j = 0; j < NF; ++j) {
            double g;
            const double fl = fma(ul[2], sy[j], fma(ul[1], cy[j], ul[0]));
            const double fm = fma(um[2], sy2[j], fma(um[1], cy2[j], um[0]));
            if (KIND == OVERLAP) {
                g = fl * fm;
            } else if (SHARED) {
                g = fl * fm * fp[32 * (i * NF + j)];
            } else {
                const double e1 = fma(B1, cy[j], A1);
                const double e2 = fma(B2, cy2[j], A2);
                g = fl * fm * bubble_F(e1, KIND == PP ? -e2 : e2, inv2T, inv4T);
            }
            rf = fma(c_wf[v][j], g, rf);
            if ((j & 1) == 0) rc = fma(c_wc[v][j >> 1], g, rc);
        }
        fine = fma(c_wf[v][i], rf, fine);
        if ((i & 1) == 0) coarse = fma(c_wc[v][i >> 1], rc, coarse);
    }
    s2 = fine;
    s1 = coarse;
}

// MONOMIAL test kind: (kx/pi)^l (ky/pi)^m; the rule is separable.
template <int N>
__device__ __forceinline__ void region_monomial(int v, uint32_t L, uint32_t ix, uint32_t iy,
                                                int a, int b, double& s2, double& s1)
{
    constexpr int NF = 2 * N + 1;
    const double hh = ldexp(1.0, -int(L));            // half side / pi
    const double xc = fma(double(2 * ix + 1), hh, -1.0), yc = fma(double(2 * iy + 1), hh, -1.0);
    double fx = 0.0, cxs = 0.0, fy = 0.0, cys = 0.0;
#pragma unroll
    for (int i = 0; i < NF; ++i) {
        const double px = pow(fma(hh, c_t[v][i], xc), double(a));
        const double py = pow(fma(hh, c_t[v][i], yc), double(b));
        fx = fma(c_wf[v][i], px, fx);
        fy = fma(c_wf[v][i], py, fy);
        if ((i & 1) == 0) {
            cxs = fma(c_wc[v][i >> 1], px, cxs);
            cys = fma(c_wc[v][i >> 1], py, cys);
        }
    }
    s2 = fx * fy;
    s1 = cxs * cys;
}

// ---------------------------------------------------------------------------
// FP32 evaluation (mixed precision).  What stays FP64: the region centre and
// node rotations, the reduced energies x = e/2T (1 DFMA each: the 1/2T factor
// is folded into the per-row coefficients) and their exact difference
// d = x1 - x2, because near the Fermi surface e is a small difference of O(1)
// terms and an FP32 energy would move x by ~1e-6 at T = 0.05; the region sums
// Q_N, Q_2N, their difference and all totals.  What runs in FP32: the
// kernel F from x1, x2, d (2 MUFU ex2 + one fast division per node), the form
// factors, and the sums of a row of nodes.
//
// Rounding noise.  Each node's FP32 value g = f_l f_m F carries independent
// rounding errors; their standard deviation, in units of 2^-24, is bounded by
//   s = kNoiseUlps |f_l f_m F|                 (ex2, products, division)
//     + 4 |F| (|f_l| + |f_m|)                   (form factors: sums of O(1) terms)
//     + |f_l f_m| dF                            (rounding x1, x2 to FP32)
// with dF = |F| (|x1| + |x2|) on the sinhc branch and
// dF = (sech^2 x1 |x1| + sech^2 x2 |x2|) / (2 |e1 - e2|) on the tanh branch
// (|dF/dx_i| |x_i| 2^-24 for F = (tanh x1 - tanh x2) / (2 (e1 - e2))).
// A region returns the rms noise of Q_N - Q_2N,
//   nse = 2^-24 (h/2)^2/(2pi)^2 sqrt(sum_ij (w_i w_j s_ij)^2 + sum_coarse (v_i v_j s_ij)^2),
// (w fine, v coarse weights).  The noise stays inside |Q_N - Q_2N| (it only
// makes the error estimate larger); an integral whose summed noise
// kNoiseSigmas * sum(nse) exceeds a quarter of its tolerance -- which no
// refinement can fix, since the sum does not shrink as regions split -- is
// re-evaluated at higher precision.
__device__ __forceinline__ float ex2_approx(float x)
{
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// F(x1, x2) with x = e/2T, d = x1 - x2 (exact), twoT = 2T, inv4T = 1/4T, in FP32,
// and dF, the sensitivity of F to rounding x1, x2 (see the noise model above).
// |d| <= 1: (1/4T) sinhc(d) sech x1 sech x2 (series of sinhc to d^10);
// |d| > 1:  the same-sign / opposite-sign forms of the FP64 kernel.
__device__ __forceinline__ float bubble_F32(float x1, float x2, float d, float twoT, float inv4T,
                                            float& dF)
{
    const float L2E = 1.4426950408889634f;
    const float a1 = fabsf(x1), a2 = fabsf(x2);
    const float v1 = ex2_approx(-a1 * L2E), v2 = ex2_approx(-a2 * L2E);
    const float u1 = v1 * v1, u2 = v2 * v2;
    const float p1 = 1.0f + u1, p2 = 1.0f + u2;
    const float p = p1 * p2;
    const bool near = fabsf(d) <= 1.0f;
    const bool neg1 = x1 < 0.0f;
    const bool same = neg1 == (x2 < 0.0f);
    float far = same ? (u2 - u1) : fmaf(-u1, u2, 1.0f);
    far = neg1 ? -far : far;
    const float d2 = d * d;
    float sh = fmaf(d2, 1.0f / 39916800.0f, 1.0f / 362880.0f);
    sh = fmaf(d2, sh, 1.0f / 5040.0f);
    sh = fmaf(d2, sh, 1.0f / 120.0f);
    sh = fmaf(d2, sh, 1.0f / 6.0f);
    sh = fmaf(d2, sh, 1.0f);
    const float nearv = (4.0f * inv4T) * (v1 * v2) * sh;
    const float num = near ? nearv : far;
    const float ediff = twoT * d;   // e1 - e2
    const float den = near ? p : p * ediff;
    const float F = __fdividef(num, den);
    // sech^2 x = 4u / (1+u)^2
    const float s1 = __fdividef(4.0f * u1, p1 * p1), s2 = __fdividef(4.0f * u2, p2 * p2);
    dF = near ? fabsf(F) * (a1 + a2) : __fdividef(fmaf(s1, a1, s2 * a2), 2.0f * fabsf(ediff));
    return F;
}

template <int N, int KIND, bool SHARED = false>
__device__ __forceinline__ void region_trig_fp32(int v, uint32_t L, uint32_t ix, uint32_t iy,
                                                 QTrig tq, int l, int m, const DevBatch& B,
                                                 Lattice lat, double& s2, double& s1, float& nz,
                                                 const float2* fp = nullptr)
{
    constexpr int NF = 2 * N + 1;
    const double inv2T = B.inv2T;
    const float twoT = float(2.0 * B.T), inv4T = float(B.inv4T);
    double sxc, cxc, syc, cyc;
    sincospi(fma(double(2 * ix + 1), ldexp(1.0, -int(L)), -1.0), &sxc, &cxc);
    sincospi(fma(double(2 * iy + 1), ldexp(1.0, -int(L)), -1.0), &syc, &cyc);

    double cyd[NF], cy2d[NF];
    float cyf[NF], syf[NF], cy2f[NF], sy2f[NF];
#pragma unroll
    for (int j = 0; j < NF; ++j) {
        const int jj = j <= N ? j : 2 * N - j;
        const double co = c_co[v][L][jj];
        const double so = j <= N ? c_so[v][L][jj] : -c_so[v][L][jj];
        const double c = fma(cyc, co, -syc * so);
        const double sn = fma(syc, co, cyc * so);
        double c2, s2_;
        if (KIND == PP) { c2 = fma(tq.cqy, c, tq.sqy * sn); s2_ = fma(tq.sqy, c, -tq.cqy * sn); }
        else            { c2 = fma(c, tq.cqy, -sn * tq.sqy); s2_ = fma(sn, tq.cqy, c * tq.sqy); }
        cyd[j] = c;
        cy2d[j] = c2;
        cyf[j] = float(c);
        syf[j] = float(sn);
        cy2f[j] = float(c2);
        sy2f[j] = float(s2_);
    }
    float Cl[3][3], Cm[3][3];
#pragma unroll
    for (int a = 0; a < 3; ++a)
#pragma unroll
        for (int b = 0; b < 3; ++b) { Cl[a][b] = c_ff32[l][a][b]; Cm[a][b] = c_ff32[m][a][b]; }

    // x = e / 2T = A(kx) + B(kx) cos ky with A = (-2t cx - mu)/2T, B = (-2t - 4t' cx)/2T
    const double tA = -2.0 * lat.t * inv2T, tB = -4.0 * lat.tp * inv2T, mu = lat.mu * inv2T;
    double fine = 0.0, coarse = 0.0;
    float noise = 0.0f;
#pragma unroll 1
    for (int i = 0; i < NF; ++i) {
        const int ii = i <= N ? i : 2 * N - i;
        const double co = c_co[v][L][ii];
        const double so = i <= N ? c_so[v][L][ii] : -c_so[v][L][ii];
        const double cx = fma(cxc, co, -sxc * so);
        const double sx = fma(sxc, co, cxc * so);
        double cx2, sx2;
        if (KIND == PP) { cx2 = fma(tq.cqx, cx, tq.sqx * sx); sx2 = fma(tq.sqx, cx, -tq.cqx * sx); }
        else            { cx2 = fma(cx, tq.cqx, -sx * tq.sqx); sx2 = fma(sx, tq.cqx, cx * tq.sqx); }
        const double A1 = fma(tA, cx, -mu), B1 = fma(tB, cx, tA);
        const double A2 = fma(tA, cx2, -mu), B2 = fma(tB, cx2, tA);
        const float cxf = float(cx), sxf = float(sx), cx2f = float(cx2), sx2f = float(sx2);
        float ul[3], um[3];
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            ul[b] = fmaf(Cl[2][b], sxf, fmaf(Cl[1][b], cxf, Cl[0][b]));
            um[b] = fmaf(Cm[2][b], sx2f, fmaf(Cm[1][b], cx2f, Cm[0][b]));
        }
        float rf = 0.0f, rc = 0.0f, rnf = 0.0f, rnc = 0.0f;
#pragma unroll
        for (int j = 0; j < NF; ++j) {
            float F, dF;
            if (SHARED) {
                const float2 f = fp[32 * (i * NF + j)];   // F and its sensitivity
                F = f.x;
                dF = f.y;
            } else {
                const double x1 = fma(B1, cyd[j], A1);
                double x2 = fma(B2, cy2d[j], A2);
                if (KIND == PP) x2 = -x2;
                F = bubble_F32(float(x1), float(x2), float(x1 - x2), twoT, inv4T, dF);
            }
            const float fl = fmaf(ul[2], syf[j], fmaf(ul[1], cyf[j], ul[0]));
            const float fm = fmaf(um[2], sy2f[j], fmaf(um[1], cy2f[j], um[0]));
            const float flm = fl * fm;
            const float g = flm * F;
            rf = fmaf(c_wf32[v][j], g, rf);
            if ((j & 1) == 0) rc = fmaf(c_wc32[v][j >> 1], g, rc);
            const float sg = fmaf(fabsf(flm), fmaf(kNoiseUlps, fabsf(F), dF),
                                  4.0f * fabsf(F) * (fabsf(fl) + fabsf(fm)));
            const float sf = c_wf32[v][j] * sg;
            rnf = fmaf(sf, sf, rnf);
            if ((j & 1) == 0) { const float sc = c_wc32[v][j >> 1] * sg; rnc = fmaf(sc, sc, rnc); }
        }
        fine = fma(c_wf[v][i], double(rf), fine);
        if ((i & 1) == 0) {
            coarse = fma(c_wc[v][i >> 1], double(rc), coarse);
            noise = fmaf(c_wc32[v][i >> 1] * c_wc32[v][i >> 1], rnc, noise);
        }
        noise = fmaf(c_wf32[v][i] * c_wf32[v][i], rnf, noise);
    }
    s2 = fine;
    s1 = coarse;
    nz = noise;
}

// ---------------------------------------------------------------------------
// Float-float ("df32") evaluation: every quantity is an unevaluated sum
// hi + lo of two FP32 numbers (about 48 significant bits), so the whole
// integrand runs on the FP32 pipe -- 64x the FP64 pipe on this GPU -- at
// close to FP64 accuracy.  Integrals whose FP32 rounding noise is too large
// for their tolerance (those that vanish by symmetry, mostly) are evaluated
// this way.  Building blocks, written from the published error-free
// transformations: Knuth's TwoSum, the FMA form of Dekker's TwoProduct, and
// the double-word add / multiply / divide of Hida, Li and Bailey's
// double-double arithmetic transposed to FP32 pairs.  Additions use the
// "sloppy" form (absolute error ~2^-48 of the operands), which is enough
// here: every sum is either of O(1) bounded terms or bounded away from
// cancellation (|d| > 1/8 on the tanh branch).
struct f2 {
    float hi, lo;
};

__device__ __forceinline__ f2 two_sum(float a, float b)
{
    const float s = a + b;
    const float bb = s - a;
    return {s, (a - (s - bb)) + (b - bb)};
}
__device__ __forceinline__ f2 fast_two_sum(float a, float b)
{
    const float s = a + b;
    return {s, b - (s - a)};
}
__device__ __forceinline__ f2 df_add(f2 a, f2 b)
{
    f2 s = two_sum(a.hi, b.hi);
    s.lo += a.lo + b.lo;
    return fast_two_sum(s.hi, s.lo);
}
__device__ __forceinline__ f2 df_add_f(f2 a, float b)
{
    f2 s = two_sum(a.hi, b);
    s.lo += a.lo;
    return fast_two_sum(s.hi, s.lo);
}
__device__ __forceinline__ f2 df_neg(f2 a) { return {-a.hi, -a.lo}; }
__device__ __forceinline__ f2 df_mul(f2 a, f2 b)
{
    const float p = a.hi * b.hi;
    float e = fmaf(a.hi, b.hi, -p);
    e = fmaf(a.hi, b.lo, e);
    e = fmaf(a.lo, b.hi, e);
    return fast_two_sum(p, e);
}
__device__ __forceinline__ f2 df_mul_f(f2 a, float b)
{
    const float p = a.hi * b;
    float e = fmaf(a.hi, b, -p);
    e = fmaf(a.lo, b, e);
    return fast_two_sum(p, e);
}
__device__ __forceinline__ float rcp_approx(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}
// a / b: a first quotient from the approximate reciprocal, one correction
// from the exact residual a - q1 b.
__device__ __forceinline__ f2 df_div(f2 a, f2 b)
{
    const float r = rcp_approx(b.hi);
    const float q1 = a.hi * r;
    const f2 res = df_add(a, df_neg(df_mul_f(b, q1)));
    const float q2 = res.hi * r;
    return fast_two_sum(q1, q2);
}
__device__ __forceinline__ f2 df_from(double x)
{
    const float hi = float(x);
    return {hi, float(x - double(hi))};
}
__device__ __forceinline__ f2 df_c(float2 c) { return {c.x, c.y}; }

// exp(-a), a >= 0, in float-float (Tang's table-driven method): k = rint(64 a / ln 2),
// r = a - k ln2/64 with ln2/64 split in three parts so that k * C1 is exact
// (k < 2^14, C1 has 10 significant bits), e^-a = 2^(-k/64) e^-r with the
// table 2^(j/64) and a degree-5 Taylor polynomial of e^-r on |r| <= ln2/128
// (truncation below 4e-17).  Results below 2^-126 are flushed to zero.
__device__ __forceinline__ f2 df_exp_neg(f2 a, const float2* tab)
{
    if (a.hi > 87.0f) return {0.0f, 0.0f};
    const float C1 = 0.010833740234375f;          // 0x1.63p-7
    const float C2 = -3.3155381515825866e-06f;
    const float C3 = 2.572804640231345e-14f;
    // k = rint(64 a_hi / ln2) by the shift 1.5 * 2^23 (a_hi 64/ln2 < 2^13):
    // the low encoding bits of the sum are k
    const float kt = fmaf(a.hi, 92.33248138427734f, 12582912.0f);
    const float k = __fsub_rn(kt, 12582912.0f);
    const float t1 = fmaf(-k, C1, a.hi);          // exact (Sterbenz)
    f2 r = two_sum(t1, a.lo);
    const f2 kc2 = {k * C2, fmaf(k, C2, -k * C2)};
    r = df_add(r, df_neg(kc2));
    r = df_add_f(r, -k * C3);
    const f2 t = df_neg(r);                       // e^-a = 2^(-k/64) e^t
    float p = fmaf(t.hi, 1.0f / 120.0f, 1.0f / 24.0f);
    p = fmaf(t.hi, p, 1.0f / 6.0f);               // 1/6 + t/24 + t^2/120
    f2 P = df_add_f(df_mul_f(t, p), 0.5f);
    P = df_add_f(df_mul(t, P), 1.0f);
    P = df_add_f(df_mul(t, P), 1.0f);
    const int n = 0x4B400000 - __float_as_int(kt);   // -k
    const int m = n >> 6;                         // floor(n / 64)
    const int j = n & 63;
    f2 res = df_mul(P, df_c(tab[j]));
    if (m < -125) return {0.0f, 0.0f};
    const float sc = __int_as_float((m + 127) << 23);
    res.hi *= sc;
    res.lo *= sc;
    return res;
}

// F(x1, x2) = [tanh x1 - tanh x2] / (2 (e1 - e2)) in float-float, x = e / 2T,
// d = x1 - x2; |d| <= 1/8: (1/4T) sinhc(d) sech x1 sech x2; else the
// same-sign / opposite-sign forms of the FP64 kernel.
__device__ __forceinline__ f2 bubble_Fdf(f2 x1, f2 x2, f2 d, f2 twoT, f2 inv4T,
                                         const float2* tab)
{
    const bool neg1 = x1.hi < 0.0f, neg2 = x2.hi < 0.0f;
    const f2 a1 = neg1 ? df_neg(x1) : x1, a2 = neg2 ? df_neg(x2) : x2;
    const f2 v1 = df_exp_neg(a1, tab), v2 = df_exp_neg(a2, tab);
    const f2 u1 = df_mul(v1, v1), u2 = df_mul(v2, v2);
    const f2 p = df_mul(df_add_f(u1, 1.0f), df_add_f(u2, 1.0f));
    f2 num, den;
    if (fabsf(d.hi) <= 0.125f) {
        // sinhc(d) = 1 + d^2/6 + d^4/120 + d^6/5040 + d^8/362880 (+ < 3e-17 at |d| = 1/8)
        const f2 d2 = df_mul(d, d);
        const float q = fmaf(d2.hi, fmaf(d2.hi, 1.0f / 362880.0f, 1.0f / 5040.0f), 1.0f / 120.0f);
        f2 S = df_add(df_mul_f(d2, q), f2{0.1666666716337204f, -4.967053879312289e-09f});
        S = df_add_f(df_mul(d2, S), 1.0f);
        num = df_mul(df_mul(df_mul_f(inv4T, 4.0f), df_mul(v1, v2)), S);
        den = p;
    } else {
        num = (neg1 == neg2) ? df_add(u2, df_neg(u1)) : df_add_f(df_neg(df_mul(u1, u2)), 1.0f);
        if (neg1) num = df_neg(num);
        den = df_mul(p, df_mul(d, twoT));   // (e1 - e2) = 2T d
    }
    return df_div(num, den);
}

// Column values of a region: cos/sin of ky and of the shifted ky (4 x NF
// float-float numbers).  Kept in registers, or (SMEM) in a shared-memory
// slice at ys[(f NF + j) kYsStride] (thread-minor, bank-conflict free),
// which frees 72 registers and lets more warps hide the latency of the
// float-float dependency chains.
constexpr int kYsStride = 128;   // threads per block of the float-float kernel

template <int NF, bool SMEM>
struct YCols {
    float2* ys;                  // shared slice (SMEM)
    f2 r[4][SMEM ? 1 : NF];      // registers otherwise
    __device__ __forceinline__ void set(int f, int j, f2 v)
    {
        if (SMEM) ys[(f * NF + j) * kYsStride] = make_float2(v.hi, v.lo);
        else r[f][SMEM ? 0 : j] = v;
    }
    __device__ __forceinline__ f2 get(int f, int j) const
    {
        if (SMEM) { const float2 t = ys[(f * NF + j) * kYsStride]; return {t.x, t.y}; }
        return r[f][SMEM ? 0 : j];
    }
};

template <int N, int KIND, bool SMEM, bool SHARED = false>
__device__ __forceinline__ void region_trig_df(int v, uint32_t L, uint32_t ix, uint32_t iy,
                                               QTrig tq, int l, int m, const DevBatch& B,
                                               Lattice lat, const float2* tab, float2* ys,
                                               double& s2, double& s1, const float2* fp = nullptr)
{
    constexpr int NF = 2 * N + 1;
    const double inv2T = B.inv2T;
    const f2 twoT = df_from(2.0 * B.T);
    const f2 inv4T = df_from(B.inv4T);
    // FP64 only for the exact dyadic centre; rotations, energies and form
    // factors below are float-float
    double sxc_, cxc_, syc_, cyc_;
    sincospi(fma(double(2 * ix + 1), ldexp(1.0, -int(L)), -1.0), &sxc_, &cxc_);
    sincospi(fma(double(2 * iy + 1), ldexp(1.0, -int(L)), -1.0), &syc_, &cyc_);
    const f2 cxc = df_from(cxc_), sxc = df_from(sxc_), cyc = df_from(cyc_), syc = df_from(syc_);
    const f2 cqx = df_from(tq.cqx), sqx = df_from(tq.sqx), cqy = df_from(tq.cqy), sqy = df_from(tq.sqy);

    YCols<NF, SMEM> Y;
    Y.ys = ys;
#pragma unroll(SHARED ? 1 : NF)
    for (int j = 0; j < NF; ++j) {
        const int jj = j <= N ? j : 2 * N - j;
        const f2 co = df_c(c_codf[v][L][jj]);
        const f2 so = j <= N ? df_c(c_sodf[v][L][jj]) : df_neg(df_c(c_sodf[v][L][jj]));
        const f2 c = df_add(df_mul(cyc, co), df_neg(df_mul(syc, so)));
        const f2 sn = df_add(df_mul(syc, co), df_mul(cyc, so));
        f2 c2, s2_;
        if (KIND == PP) {   // q - k
            c2 = df_add(df_mul(cqy, c), df_mul(sqy, sn));
            s2_ = df_add(df_mul(sqy, c), df_neg(df_mul(cqy, sn)));
        } else {            // k + q
            c2 = df_add(df_mul(c, cqy), df_neg(df_mul(sn, sqy)));
            s2_ = df_add(df_mul(sn, cqy), df_mul(c, sqy));
        }
        Y.set(0, j, c);
        Y.set(1, j, sn);
        Y.set(2, j, c2);
        Y.set(3, j, s2_);
    }
    // x = e / 2T = A(kx) + B(kx) cos ky, A = -(2t cx + mu)/2T, B = -(2t + 4t' cx)/2T
    const f2 tA = df_from(-2.0 * lat.t * inv2T), tB = df_from(-4.0 * lat.tp * inv2T);
    const f2 nmu = df_from(-lat.mu * inv2T);
    double fine = 0.0, coarse = 0.0;
#pragma unroll 1
    for (int i = 0; i < NF; ++i) {
        const int ii = i <= N ? i : 2 * N - i;
        const f2 co = df_c(c_codf[v][L][ii]);
        const f2 so = i <= N ? df_c(c_sodf[v][L][ii]) : df_neg(df_c(c_sodf[v][L][ii]));
        const f2 cx = df_add(df_mul(cxc, co), df_neg(df_mul(sxc, so)));
        const f2 sx = df_add(df_mul(sxc, co), df_mul(cxc, so));
        f2 cx2, sx2;
        if (KIND == PP) {
            cx2 = df_add(df_mul(cqx, cx), df_mul(sqx, sx));
            sx2 = df_add(df_mul(sqx, cx), df_neg(df_mul(cqx, sx)));
        } else {
            cx2 = df_add(df_mul(cx, cqx), df_neg(df_mul(sx, sqx)));
            sx2 = df_add(df_mul(sx, cqx), df_mul(cx, sqx));
        }
        const f2 A1 = df_add(df_mul(tA, cx), nmu), B1 = df_add(df_mul(tB, cx), tA);
        const f2 A2 = df_add(df_mul(tA, cx2), nmu), B2 = df_add(df_mul(tB, cx2), tA);
        f2 ul[3], um[3];
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            ul[b] = df_add(df_add(df_mul(df_c(c_ffdf[l][1][b]), cx), df_mul(df_c(c_ffdf[l][2][b]), sx)),
                           df_c(c_ffdf[l][0][b]));
            um[b] = df_add(df_add(df_mul(df_c(c_ffdf[m][1][b]), cx2), df_mul(df_c(c_ffdf[m][2][b]), sx2)),
                           df_c(c_ffdf[m][0][b]));
        }
        f2 rf = {0.0f, 0.0f}, rc = {0.0f, 0.0f};
        // with F read from the tables two columns a trip: fully unrolled it spills 680
        // bytes at 128 registers (10.9 ms on 4,050 integrals with N = 6; two columns
        // 6.9, one 8.8, four 7.1)
        constexpr int kUnroll = SHARED ? 2 : NF;
#pragma unroll(kUnroll)
        for (int j = 0; j < NF; ++j) {
            const f2 cyj = Y.get(0, j), syj = Y.get(1, j), cy2j = Y.get(2, j), sy2j = Y.get(3, j);
            f2 F;
            if (SHARED) {
                F = df_c(fp[32 * (i * NF + j)]);
            } else {
                const f2 x1 = df_add(df_mul(B1, cyj), A1);
                f2 x2 = df_add(df_mul(B2, cy2j), A2);
                if (KIND == PP) x2 = df_neg(x2);
                F = bubble_Fdf(x1, x2, df_add(x1, df_neg(x2)), twoT, inv4T, tab);
            }
            const f2 fl = df_add(df_add(df_mul(ul[1], cyj), df_mul(ul[2], syj)), ul[0]);
            const f2 fm = df_add(df_add(df_mul(um[1], cy2j), df_mul(um[2], sy2j)), um[0]);
            const f2 g = df_mul(df_mul(fl, fm), F);
            rf = df_add(rf, df_mul(df_c(c_wfdf[v][j]), g));
            if ((j & 1) == 0) rc = df_add(rc, df_mul(df_c(c_wcdf[v][j >> 1]), g));
        }
        fine = fma(c_wf[v][i], double(rf.hi) + double(rf.lo), fine);
        if ((i & 1) == 0) coarse = fma(c_wc[v][i >> 1], double(rc.hi) + double(rc.lo), coarse);
    }
    s2 = fine;
    s1 = coarse;
}

// PH / PP regions of integrals escalated to float-float (and not set to FP64).
__device__ __forceinline__ bool is_df_region(uint32_t mt)
{
    const int kind = meta_kind(mt);
    return meta_valid(mt) && (mt & kMetaDf32) != 0u && (mt & kMetaFp64) == 0u &&
           (kind == PH || kind == PP);
}

// ---------------------------------------------------------------------------
// The kernel F shared between integrals.  F at a region's nodes depends on (kind, T,
// q) and the region, not on the form factors, and the partitions of the (l, m) pairs
// of one q overlap: of the regions a round evaluates, most keys occur for several
// pairs of a q (18 times each on average for 81 pairs at T = 0.05).  Before the
// evaluation, one pass finds the distinct (q, region, precision) entries with a hash
// table, a second evaluates F once for each of them, a thread per row of nodes (which
// also keeps a round of few regions short: a thread per region needs 90 us for one),
// and the evaluation reads F where it would compute it.  F takes 65 of a node's 75
// FP64 instructions and 300 of its 400 float-float ones.
//
// The tables live in the pool buffers that the round's split has not written yet:
// hash slots in err[next], per entry its distinct index or the entry that holds it
// in nse[next], per distinct index an entry in key[next], F in val[next] and the rest
// of key[next], in blocks of 32 regions [node][region].  A distinct region without
// room, or an entry whose probes run out, is evaluated as before.
//
// Reading F pays where enough entries share it, so once the distinct entries are
// counted the round decides for each class.  One round, T = 0.1, whole call with the
// tables / without, p entries per distinct one:
//   entries       1,024  16,384  65,536  262,144  1,048,576
//   FP64  p = 1    0.53   0.68    1.00    1.10    1.12   (N = 6: 0.41 ... 1.17)
//         p = 2    0.50   0.56    0.64    0.65    0.65
//   FP32  p = 1    0.95   1.07    1.26    1.40    1.49   (N = 6: 0.82 ... 1.43)
//         p = 2    0.93   1.00    1.00    0.99    0.97   (N = 6: 0.77 ... 0.87)
//         p = 3    0.91   0.94    0.92    0.84    0.79
//   float-float
//         p = 1    0.84   1.06    1.07    1.21    1.22   (N = 6: 0.69 ... 1.13)
//         p = 2    0.85   0.94    0.88    0.83    0.79
// (small rounds gain without repeats, from the thread per row of nodes).  Which calls
// count at all: shares_kernel.
constexpr uint32_t kNoShare = 0xffffffffu, kShareRef = 0x80000000u;
constexpr int kShareProbes = 32;
constexpr int64_t kShareMax = int64_t(1) << 30;   // entries of a round

struct Share {
    uint32_t* slot;            // hash table: entry + 1, or 0
    uint64_t mask;             // its size - 1 (a power of two)
    uint32_t* uid;             // per entry: distinct index, kShareRef | entry, or kNoShare
    uint32_t* rep;             // per distinct index: an entry
    double *f0, *f1;           // F blocks (f1 after nf0 of them)
    uint32_t nf0, room;        // blocks in f0; distinct indices with room for F
};

__device__ __forceinline__ Share share_view(const Work& w, int nodes)
{
    const int nxt = w.ls->cur ^ 1;
    const int64_t n = w.ls->n_eval, block = 32 * int64_t(nodes);
    Share s;
    uint64_t size = 1;
    while (size < uint64_t(2 * n)) size <<= 1;
    while (size > uint64_t(2 * w.cap)) size >>= 1;
    s.slot = reinterpret_cast<uint32_t*>(w.err[nxt]);
    s.mask = size - 1;
    s.uid = reinterpret_cast<uint32_t*>(w.nse[nxt]);
    s.rep = reinterpret_cast<uint32_t*>(w.key[nxt]);
    s.f0 = w.val[nxt];
    s.nf0 = uint32_t(w.cap / block);
    const int64_t used = (n + 63) / 64 * 32;   // doubles of key[next] that rep takes
    s.f1 = reinterpret_cast<double*>(w.key[nxt]) + used;
    const int64_t nf1 = w.cap > used ? (w.cap - used) / block : 0;
    s.room = uint32_t(min(int64_t(s.nf0) + nf1, kShareMax / 32) * 32);
    return s;
}
__device__ __forceinline__ bool sharing(const Work& w, int64_t n)
{
    return w.share && n > 0 && n < kShareMax;
}
// The counts of a round after k_share_insert or k_first_insert, loaded together (one
// after the other they cost every kernel that asks half a microsecond).
struct RoundCounts {
    int64_t n;
    unsigned long long distinct, sharable, unshared;
};
__device__ __forceinline__ RoundCounts round_counts(const Work& w)
{
    const RoundTotals& t = *w.totals;
    const int64_t n = w.ls->n_eval;
    const unsigned long long distinct = t.distinct, other = t.unsharable, unshared = t.unshared;
    return {n, distinct, (unsigned long long)n - other, unshared};
}
// whether the round reads F of a class (0 FP64, 1 FP32, 2 float-float) from the tables:
// in small rounds, and where the distinct entries are few enough of those that could
// share; with half of them at least in the tables
template <int N, int CLASS>
__device__ __forceinline__ bool share_used(const RoundCounts& r, const Share& s)
{
    constexpr int64_t small = CLASS == 0 || N > 4 ? 32768 : 8192;
    constexpr unsigned long long eighths =
        CLASS == 0 ? 7 : CLASS == 1 ? (N > 4 ? 5 : 4) : (N > 4 ? 7 : 6);
    return r.distinct <= 2ull * s.room &&
           (r.n <= small || 8 * r.distinct <= eighths * r.sharable);
}
// F of distinct region u: node k at [32 k]
__device__ __forceinline__ double* share_f(const Share& s, uint32_t u, int nodes)
{
    const uint32_t b = u >> 5;
    const size_t block = 32 * size_t(nodes);
    return (b < s.nf0 ? s.f0 + b * block : s.f1 + (b - s.nf0) * block) + (u & 31u);
}
// the distinct region of entry t, or kNoShare when it has none with room
__device__ __forceinline__ uint32_t share_find(const Share& s, int64_t t)
{
    uint32_t u = s.uid[t];
    if (u != kNoShare && (u & kShareRef)) u = s.uid[u & ~kShareRef];
    return u < s.room ? u : kNoShare;
}
// how an entry's F is evaluated: 0 FP64, 1 FP32, 2 float-float; -1 not shared
template <bool FP32>
__device__ __forceinline__ int share_class(uint32_t mt)
{
    const int kind = meta_kind(mt);
    if (!meta_valid(mt) || (kind != PH && kind != PP)) return -1;
    if (!FP32) return 0;
    return (mt & kMetaFp64) ? -1 : (mt & kMetaDf32) ? 2 : 1;
}

__global__ void k_share_clear(Work w, int nodes)
{
    if (!sharing(w, w.ls->n_eval)) return;
    const Share s = share_view(w, nodes);
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    for (uint64_t i = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x; i <= s.mask; i += stride)
        s.slot[i] = 0u;
    if (blockIdx.x == 0 && threadIdx.x == 0)
        w.totals->unsharable = w.totals->distinct = w.totals->unshared = 0ull;
}

// Whether the round's evaluation reads the tables, for paid_last_sharing: by one thread
// of the launch's last block, which has the least to do.
__device__ __forceinline__ void note_sharing(const Work& w, const RoundCounts& r, bool used,
                                             uint32_t room)
{
    if (blockIdx.x != gridDim.x - 1 || threadIdx.x != blockDim.x - 1) return;
    RoundTotals& t = *w.totals;
    if (!used) {
        t.sh_skipped += 1;
        return;
    }
    t.sh_rounds += 1;
    t.sh_entries += r.sharable;
    t.sh_distinct += r.distinct;
    t.sh_unshared += r.unshared;
    t.sh_roomless += r.distinct > room ? r.distinct - room : 0ull;
}
// a thread's entries of a round (at most kShareMax over the grid's threads, some 4,600),
// in the low half those that cannot share, in the high half those without a place, both
// mostly none (counting those that can cost 5 ns a warp, 10 us a round of 65,536)
__device__ __forceinline__ void add_left_out(const Work& w, unsigned count)
{
    if (!__any_sync(0xffffffffu, count)) return;
    const unsigned other = __reduce_add_sync(0xffffffffu, count & 0xffffu);
    const unsigned lost = __reduce_add_sync(0xffffffffu, count >> 16);
    if ((threadIdx.x & 31) == 0) {
        if (other) atomicAdd(&w.totals->unsharable, (unsigned long long)other);
        if (lost) atomicAdd(&w.totals->unshared, (unsigned long long)lost);
    }
}

template <bool FP32>
__global__ void __launch_bounds__(256) k_share_insert(Work w, int nodes)
{
    if (!sharing(w, w.ls->n_eval)) return;
    const Share s = share_view(w, nodes);
    const int cur = w.ls->cur;
    const int64_t n = w.ls->n_eval;
    const int lane = threadIdx.x & 31;
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    unsigned left_out = 0;
    for (int64_t t0 = int64_t(blockIdx.x) * blockDim.x + threadIdx.x - lane; t0 < n; t0 += stride) {
        const int64_t t = t0 + lane;
        uint32_t u = kNoShare;
        bool mine = false;
        if (t < n) {
            const uint2 e = w.evl[t];
            const uint32_t mt = w.meta[e.y];
            const int cls = share_class<FP32>(mt);
            if (cls < 0) {
                ++left_out;
            } else {
                const uint64_t key = w.key[cur][e.x];
                const DevBatch& B = w.batches[meta_batch(mt)];
                const uint32_t np = uint32_t(B.npairs);
                // the first integral of the entry's q
                const uint32_t g0 = e.y - uint32_t((int64_t(e.y) - B.first) % np);
                uint64_t h = key ^ ((uint64_t(g0) << 2 | uint64_t(cls)) * 0x9e3779b97f4a7c15ull);
                h = (h ^ (h >> 30)) * 0xbf58476d1ce4e5b9ull;   // splitmix64's finaliser
                h = (h ^ (h >> 27)) * 0x94d049bb133111ebull;
                h ^= h >> 31;
                for (int p = 0; p < kShareProbes; ++p) {
                    const uint32_t old = atomicCAS(&s.slot[(h + p) & s.mask], 0u, uint32_t(t) + 1u);
                    if (old == 0u) { mine = true; break; }
                    const uint2 o = w.evl[old - 1u];
                    if (o.y >= g0 && o.y - g0 < np && w.key[cur][o.x] == key &&
                        (!FP32 || share_class<FP32>(w.meta[o.y]) == cls)) {
                        u = kShareRef | (old - 1u);
                        break;
                    }
                }
                if (!mine && u == kNoShare) left_out += 0x10000u;   // its probes ran out
            }
        }
        // distinct indices in entry order within a warp: siblings stay together
        const unsigned m = __ballot_sync(0xffffffffu, mine);
        unsigned long long base = 0;
        if (lane == 0 && m) base = atomicAdd(&w.totals->distinct, (unsigned long long)__popc(m));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (mine) {
            u = uint32_t(base) + uint32_t(__popc(m & ((1u << lane) - 1u)));
            if (u < s.room) s.rep[u] = uint32_t(t);
        }
        if (t < n) s.uid[t] = u;
    }
    add_left_out(w, left_out);
}

// F of the distinct regions: NF threads per region, thread i owning row i and
// column i of its nodes.  Each class's arithmetic is that of its region function.
template <int N> struct ShareShape;
template <> struct ShareShape<4> { static constexpr int R = 14; };   // 126 threads
template <> struct ShareShape<6> { static constexpr int R = 9; };    // 117

template <int N, bool FP32>
__global__ void __launch_bounds__(ShareShape<N>::R * (2 * N + 1)) k_share_f(Work w, Lattice lat)
{
    constexpr int NF = 2 * N + 1, R = ShareShape<N>::R;
    __shared__ double C[R][4];                       // sin, cos of the centre (x, y) times pi
    __shared__ __align__(16) double Y[R][NF][2];     // cos ky, cos ky' (FP64, or float-float pairs)
    __shared__ float2 tab[64];
    const RoundCounts rc = round_counts(w);
    if (!sharing(w, rc.n)) return;
    const Share s = share_view(w, NF * NF);
    const bool use1 = share_used<N, FP32 ? 1 : 0>(rc, s);   // the FP32 or FP64 class
    const bool use2 = FP32 && share_used<N, 2>(rc, s);      // float-float
    note_sharing(w, rc, use1 || use2, s.room);
    if (!use1 && !use2) return;
    const int cur = w.ls->cur;
    const uint32_t count = uint32_t(min((unsigned long long)s.room, rc.distinct));
    const int rho = threadIdx.x / NF, i = threadIdx.x % NF, v = rule_variant(N);
    if (FP32)
        for (int k = threadIdx.x; k < 64; k += blockDim.x) tab[k] = c_exp2tab[k];
    for (uint32_t u0 = blockIdx.x * R; u0 < count; u0 += gridDim.x * R) {
        const uint32_t u = u0 + rho;
        bool live = u < count;
        uint32_t L = 0, g = 0;
        if (live) {
            const uint2 e = w.evl[s.rep[u]];
            g = e.y;
            if (FP32) live = share_class<true>(w.meta[g]) == 1 ? use1 : use2;
            const uint64_t key = w.key[cur][e.x];
            L = key_level(key);
            if (i < 2) {   // the exact dyadic centre / pi: -1 + (2 ix + 1) 2^-L, x then y
                const uint32_t ic = i == 0 ? key_ix(key) : key_iy(key);
                sincospi(fma(double(2 * ic + 1), ldexp(1.0, -int(L)), -1.0), &C[rho][2 * i],
                         &C[rho][2 * i + 1]);
            }
        }
        __syncthreads();
        uint32_t mt = 0;
        int cls = 0;
        bool pp = false;
        const DevBatch* B = nullptr;
        const int ii = i <= N ? i : 2 * N - i;
        double A1 = 0.0, B1 = 0.0, A2 = 0.0, B2 = 0.0;
        f2 a1 = {0.0f, 0.0f}, b1 = a1, a2 = a1, b2 = a1;
        if (live) {
            mt = w.meta[g];
            cls = share_class<FP32>(mt);
            pp = meta_kind(mt) == PP;
            B = &w.batches[meta_batch(mt)];
            const QTrig tq = w.trig[g];
            if (!FP32 || cls == 1) {
                const double co = c_co[v][L][ii];
                const double so = i <= N ? c_so[v][L][ii] : -c_so[v][L][ii];
                const double sxc = C[rho][0], cxc = C[rho][1], syc = C[rho][2], cyc = C[rho][3];
                const double cx = fma(cxc, co, -sxc * so), sx = fma(sxc, co, cxc * so);
                const double cy = fma(cyc, co, -syc * so), sy = fma(syc, co, cyc * so);
                const double cx2 = pp ? fma(tq.cqx, cx, tq.sqx * sx) : fma(cx, tq.cqx, -sx * tq.sqx);
                const double cy2 = pp ? fma(tq.cqy, cy, tq.sqy * sy) : fma(cy, tq.cqy, -sy * tq.sqy);
                Y[rho][i][0] = cy;
                Y[rho][i][1] = cy2;
                // e = A + B cos ky along the row (FP32: in units of 2T)
                const double h = FP32 ? B->inv2T : 1.0;
                const double tA = -2.0 * lat.t * h, tB = -4.0 * lat.tp * h, mu = lat.mu * h;
                A1 = fma(tA, cx, -mu);
                B1 = fma(tB, cx, tA);
                A2 = fma(tA, cx2, -mu);
                B2 = fma(tB, cx2, tA);
            } else {
                const f2 cqx = df_from(tq.cqx), sqx = df_from(tq.sqx);
                const f2 cqy = df_from(tq.cqy), sqy = df_from(tq.sqy);
                const f2 co = df_c(c_codf[v][L][ii]);
                const f2 so = i <= N ? df_c(c_sodf[v][L][ii]) : df_neg(df_c(c_sodf[v][L][ii]));
                const f2 sxc = df_from(C[rho][0]), cxc = df_from(C[rho][1]);
                const f2 syc = df_from(C[rho][2]), cyc = df_from(C[rho][3]);
                const f2 cx = df_add(df_mul(cxc, co), df_neg(df_mul(sxc, so)));
                const f2 sx = df_add(df_mul(sxc, co), df_mul(cxc, so));
                const f2 cy = df_add(df_mul(cyc, co), df_neg(df_mul(syc, so)));
                const f2 sy = df_add(df_mul(syc, co), df_mul(cyc, so));
                const f2 cx2 = pp ? df_add(df_mul(cqx, cx), df_mul(sqx, sx))
                                  : df_add(df_mul(cx, cqx), df_neg(df_mul(sx, sqx)));
                const f2 cy2 = pp ? df_add(df_mul(cqy, cy), df_mul(sqy, sy))
                                  : df_add(df_mul(cy, cqy), df_neg(df_mul(sy, sqy)));
                float2* y = reinterpret_cast<float2*>(Y[rho][i]);
                y[0] = make_float2(cy.hi, cy.lo);
                y[1] = make_float2(cy2.hi, cy2.lo);
                const f2 tA = df_from(-2.0 * lat.t * B->inv2T), tB = df_from(-4.0 * lat.tp * B->inv2T);
                const f2 nmu = df_from(-lat.mu * B->inv2T);
                a1 = df_add(df_mul(tA, cx), nmu);
                b1 = df_add(df_mul(tB, cx), tA);
                a2 = df_add(df_mul(tA, cx2), nmu);
                b2 = df_add(df_mul(tB, cx2), tA);
            }
        }
        __syncthreads();
        if (live) {
            double* f = share_f(s, u, NF * NF) + 32 * size_t(i * NF);
            if (!FP32) {
#pragma unroll 1
                for (int j = 0; j < NF; ++j) {
                    const double e1 = fma(B1, Y[rho][j][0], A1);
                    const double e2 = fma(B2, Y[rho][j][1], A2);
                    f[32 * j] = bubble_F(e1, pp ? -e2 : e2, B->inv2T, B->inv4T);
                }
            } else if (cls == 1) {
                const float twoT = float(2.0 * B->T), inv4T = float(B->inv4T);
#pragma unroll 1
                for (int j = 0; j < NF; ++j) {
                    const double x1 = fma(B1, Y[rho][j][0], A1);
                    double x2 = fma(B2, Y[rho][j][1], A2);
                    if (pp) x2 = -x2;
                    float dF;
                    const float F = bubble_F32(float(x1), float(x2), float(x1 - x2), twoT, inv4T, dF);
                    *reinterpret_cast<float2*>(f + 32 * j) = make_float2(F, dF);
                }
            } else {
                const f2 twoT = df_from(2.0 * B->T), inv4T = df_from(B->inv4T);
#pragma unroll 1
                for (int j = 0; j < NF; ++j) {
                    const float2* y = reinterpret_cast<const float2*>(Y[rho][j]);
                    const f2 x1 = df_add(df_mul(b1, df_c(y[0])), a1);
                    f2 x2 = df_add(df_mul(b2, df_c(y[1])), a2);
                    if (pp) x2 = df_neg(x2);
                    const f2 F = bubble_Fdf(x1, x2, df_add(x1, df_neg(x2)), twoT, inv4T, tab);
                    *reinterpret_cast<float2*>(f + 32 * j) = make_float2(F.hi, F.lo);
                }
            }
        }
        __syncthreads();
    }
}

template <int N, bool FP32>
static void share_launch(const Work& w, int64_t hint_eval, Lattice lat, cudaStream_t s)
{
    constexpr int NF = 2 * N + 1, R = ShareShape<N>::R;
    const int64_t blocks = std::min<int64_t>((hint_eval + 255) / 256, 152 * 8);
    k_share_clear<<<int(blocks), 256, 0, s>>>(w, NF * NF);
    k_share_insert<FP32><<<int(blocks), 256, 0, s>>>(w, NF * NF);
    k_share_f<N, FP32><<<int(std::min<int64_t>((hint_eval + R - 1) / R, 152 * 16)), R * NF, 0, s>>>(
        w, lat);
}

// Float-float evaluation kernels, one region per thread.  SHARED: the regions whose
// kernel F is in the tables, the column values in a shared-memory slice per thread
// (kYsStride-minor), so that four 128-thread blocks fit per SM (one kernel with the
// columns of N = 6 in registers, beside the code for F, took 254 of them and 9.2 ms
// where this one takes 6.9).  Otherwise the regions without: the slice for N = 4,
// so that three blocks fit, registers for N = 6.
template <int N, bool SHARED>
struct DfColumns {
    static constexpr bool kSmem = SHARED || N == 4;
    static constexpr int kBytes = kSmem ? 4 * (2 * N + 1) * kYsStride * int(sizeof(float2)) : 0;
};

template <int N, bool SHARED>
__global__ void __launch_bounds__(kYsStride, SHARED ? 4 : N == 4 ? 3 : 1)
k_eval_df(Work w, Lattice lat)
{
    constexpr bool SMEM = DfColumns<N, SHARED>::kSmem;
    constexpr int NF = 2 * N + 1;
    const int cur = w.ls->cur;
    const int64_t n_eval = w.ls->n_eval;
    const int v = N == 4 ? 0 : 1;
    extern __shared__ float2 ysm[];
    __shared__ float2 tab[64];
    const RoundCounts rc = round_counts(w);
    const Share sh = sharing(w, rc.n) ? share_view(w, NF * NF) : Share{};
    const bool share = sharing(w, rc.n) && share_used<N, 2>(rc, sh);
    if (SHARED && !share) return;
    // every float-float region is in the tables
    if (!SHARED && share && rc.unshared == 0ull && rc.distinct <= sh.room) return;
    if (threadIdx.x < 64) tab[threadIdx.x] = c_exp2tab[threadIdx.x];
    __syncthreads();
    float2* ys = SMEM ? ysm + threadIdx.x : nullptr;
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    unsigned count = 0;
    for (int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; t < n_eval; t += stride) {
        const uint2 e = w.evl[t];
        const uint32_t pos = e.x, g = e.y;
        const uint32_t mt = w.meta[g];
        if (!is_df_region(mt)) continue;
        const uint32_t u = share ? share_find(sh, t) : kNoShare;
        if ((u != kNoShare) != SHARED) continue;
        ++count;
        const uint64_t key = w.key[cur][pos];
        const DevBatch& B = w.batches[meta_batch(mt)];
        const uint32_t L = key_level(key), ix = key_ix(key), iy = key_iy(key);
        const QTrig tq = w.trig[g];
        const int l = meta_l(mt), m = meta_m(mt);
        double s2, s1;
        const float2* fp = SHARED ? reinterpret_cast<const float2*>(share_f(sh, u, NF * NF)) : nullptr;
        if (meta_kind(mt) == PH)
            region_trig_df<N, PH, SMEM, SHARED>(v, L, ix, iy, tq, l, m, B, lat, tab, ys, s2, s1, fp);
        else
            region_trig_df<N, PP, SMEM, SHARED>(v, L, ix, iy, tq, l, m, B, lat, tab, ys, s2, s1, fp);
        const double scale = ldexp(0.25, -2 * int(L));
        const double q2 = s2 * scale, q1 = s1 * scale;
        w.val[cur][pos] = q2;
        w.err[cur][pos] = fabs(q1 - q2);
        w.nse[cur][pos] = 0.0f;   // ~2^-44 relative: below every accepted tolerance
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) count += __shfl_xor_sync(0xffffffffu, count, o);
    if ((threadIdx.x & 31) == 0 && count) atomicAdd(&w.totals->df_regions, (unsigned long long)count);
}

template <int N, bool SHARED>
static void df_launch(const Work& w, int64_t hint_eval, Lattice lat, cudaStream_t s)
{
    const int blocks = int(std::min<int64_t>((hint_eval + kYsStride - 1) / kYsStride, 152 * 48));
    k_eval_df<N, SHARED><<<blocks, kYsStride, DfColumns<N, SHARED>::kBytes, s>>>(w, lat);
}

// Mixed-precision evaluation: PH / PP regions use the FP32 path (regions of
// integrals escalated to float-float are left to k_eval_df); integrals set to
// FP64 and the test kinds use the FP64 path.
template <int N>
__global__ void __launch_bounds__(128) k_eval_fp32(Work w, Lattice lat)
{
    constexpr int NF = 2 * N + 1;
    const int cur = w.ls->cur;
    const int64_t n_eval = w.ls->n_eval;
    const int v = N == 4 ? 0 : 1;
    const RoundCounts rc = round_counts(w);
    const Share sh = sharing(w, rc.n) ? share_view(w, NF * NF) : Share{};
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    // a loop of its own for rounds without tables (one loop for both took 2.11 ms where
    // this one takes 1.89 on 1,048,576 regions, FP32, N = 4)
    auto regions = [&](auto shared) {
        constexpr bool SHARED = decltype(shared)::value;
        for (int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; t < n_eval; t += stride) {
            const uint2 e = w.evl[t];
            const uint32_t pos = e.x, g = e.y;
            const uint32_t mt = w.meta[g];
            if (is_df_region(mt)) continue;   // evaluated by k_eval_df
            const uint64_t key = w.key[cur][pos];
            const DevBatch& B = w.batches[meta_batch(mt)];
            const uint32_t L = key_level(key), ix = key_ix(key), iy = key_iy(key);
            const int kind = meta_kind(mt);
            double s2 = NAN, s1 = NAN;
            float nz = 0.0f;
            if (meta_valid(mt)) {
                const QTrig tq = w.trig[g];
                const int l = meta_l(mt), m = meta_m(mt);
                const bool fp64 = (mt & kMetaFp64) != 0u;
                const uint32_t u = SHARED ? share_find(sh, t) : kNoShare;
                const float2* fp = u == kNoShare
                    ? nullptr : reinterpret_cast<const float2*>(share_f(sh, u, NF * NF));
                if (SHARED && kind == PH && fp)
                    region_trig_fp32<N, PH, true>(v, L, ix, iy, tq, l, m, B, lat, s2, s1, nz, fp);
                else if (SHARED && kind == PP && fp)
                    region_trig_fp32<N, PP, true>(v, L, ix, iy, tq, l, m, B, lat, s2, s1, nz, fp);
                else if (kind == PH && !fp64)
                    region_trig_fp32<N, PH>(v, L, ix, iy, tq, l, m, B, lat, s2, s1, nz);
                else if (kind == PP && !fp64)
                    region_trig_fp32<N, PP>(v, L, ix, iy, tq, l, m, B, lat, s2, s1, nz);
                else if (kind == PH)
                    region_trig_fp64<N, PH>(v, L, ix, iy, tq, l, m, B, lat, s2, s1);
                else if (kind == PP)
                    region_trig_fp64<N, PP>(v, L, ix, iy, tq, l, m, B, lat, s2, s1);
                else if (kind == OVERLAP)
                    region_trig_fp64<N, OVERLAP>(v, L, ix, iy, tq, l, m, B, lat, s2, s1);
                else
                    region_monomial<N>(v, L, ix, iy, l, m, s2, s1);
            }
            const double scale = ldexp(0.25, -2 * int(L));
            const double q2 = s2 * scale, q1 = s1 * scale;
            w.val[cur][pos] = q2;
            w.err[cur][pos] = fabs(q1 - q2);
            // nz = sum (w_i w_j s_ij)^2: rms noise 2^-24 scale sqrt(nz)
            w.nse[cur][pos] = float(sqrt(double(nz)) * scale * 5.9604644775390625e-8);
        }
    };
    if (sharing(w, rc.n) && share_used<N, 1>(rc, sh)) regions(std::true_type());
    else regions(std::false_type());
}

template <int N>
__global__ void __launch_bounds__(128) k_eval_fp64(Work w, Lattice lat)
{
    constexpr int NF = 2 * N + 1;
    const int cur = w.ls->cur;
    const int64_t n_eval = w.ls->n_eval;
    const int v = N == 4 ? 0 : 1;
    const RoundCounts rc = round_counts(w);
    const Share sh = sharing(w, rc.n) ? share_view(w, NF * NF) : Share{};
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    auto regions = [&](auto shared) {
        constexpr bool SHARED = decltype(shared)::value;
        for (int64_t t = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; t < n_eval; t += stride) {
            const uint2 e = w.evl[t];
            const uint32_t pos = e.x, g = e.y;
            const uint64_t key = w.key[cur][pos];
            const uint32_t mt = w.meta[g];
            const DevBatch& B = w.batches[meta_batch(mt)];
            const uint32_t L = key_level(key), ix = key_ix(key), iy = key_iy(key);
            const int kind = meta_kind(mt);
            double s2 = NAN, s1 = NAN;
            if (meta_valid(mt)) {
                const QTrig tq = w.trig[g];
                const int l = meta_l(mt), m = meta_m(mt);
                const uint32_t u = SHARED ? share_find(sh, t) : kNoShare;
                const double* fp = u == kNoShare ? nullptr : share_f(sh, u, NF * NF);
                if (SHARED && kind == PH && fp)
                    region_trig_fp64<N, PH, true>(v, L, ix, iy, tq, l, m, B, lat, s2, s1, fp);
                else if (SHARED && kind == PP && fp)
                    region_trig_fp64<N, PP, true>(v, L, ix, iy, tq, l, m, B, lat, s2, s1, fp);
                else if (kind == PH)
                    region_trig_fp64<N, PH>(v, L, ix, iy, tq, l, m, B, lat, s2, s1);
                else if (kind == PP)
                    region_trig_fp64<N, PP>(v, L, ix, iy, tq, l, m, B, lat, s2, s1);
                else if (kind == OVERLAP)
                    region_trig_fp64<N, OVERLAP>(v, L, ix, iy, tq, l, m, B, lat, s2, s1);
                else
                    region_monomial<N>(v, L, ix, iy, l, m, s2, s1);
            }
            // (h/2)^2 / (2 pi)^2 with h = 2 pi 2^-L:  2^-2L / 4
            const double scale = ldexp(0.25, -2 * int(L));
            const double q2 = s2 * scale, q1 = s1 * scale;
            w.val[cur][pos] = q2;
            w.err[cur][pos] = fabs(q1 - q2);
            w.nse[cur][pos] = 0.0f;
        }
    };
    if (sharing(w, rc.n) && share_used<N, 0>(rc, sh)) regions(std::true_type());
    else regions(std::false_type());
}

// ---------------------------------------------------------------------------
// FP64 exp and division of the shared-partition kernel.
//
// exp(-a), a >= 0: P. T. P. Tang's table-driven method (ACM TOMS 15, 1989):
// -a = n ln2/64 + r with n = round(-a 64/ln2) = 64 m + j, 0 <= j < 64, so
// exp(-a) = 2^m 2^(j/64) exp(r), |r| <= ln2/128.  r comes from a two-constant
// Cody-Waite reduction (L1 = ln2/64 to 32 significant bits, so n L1 is exact
// for |n| < 2^21; L2 = ln2/64 - L1), exp(r) from its degree-5 Taylor
// polynomial (truncation r^6/720 < 2^-54 on that interval) and 2^(j/64) from a
// 64-entry table; 2^m enters as an integer add to the exponent field.  Results
// below 2^-1022 flush to zero; NaN propagates.
__device__ __forceinline__ double exp_neg(double a, const double* tab)
{
    a = a > 800.0 ? 800.0 : a;
    const double n = rint(a * -92.33248261689366);
    double r = fma(n, -0x1.62e42ffp-7, -a);
    r = fma(n, 0x1.718432a1b0e26p-41, r);
    double p = fma(r, 1.0 / 120.0, 1.0 / 24.0);
    p = fma(r, p, 1.0 / 6.0);
    p = fma(r, p, 0.5);
    p = fma(r, p, 1.0);
    p = fma(r, p, 1.0);
    const int ni = int(n);
    const int m = ni >> 6;          // floor(n / 64)
    const int j = ni & 63;
    const double y = tab[j] * p;    // in [0.99, 2.02]: exponent field 1022 ... 1024
    const long long b = __double_as_longlong(y) + ((long long)m << 52);
    if (y != y) return y;           // NaN in, NaN out (the integer n of a NaN is arbitrary)
    return (m >= -1022 && (b >> 52) > 0) ? __longlong_as_double(b) : 0.0;
}

// num / den for a normal, non-zero den: the approximate FP64 reciprocal of
// the PTX ISA (rcp.approx.ftz.f64) refined by two Newton-Raphson steps
// y <- y + y (1 - den y), then one residual correction of the quotient
// q <- q + (num - den q) y.
__device__ __forceinline__ double div_nr(double num, double den)
{
    double y;
    asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(y) : "d"(den));
    double e = fma(-den, y, 1.0);
    y = fma(y, e, y);
    e = fma(-den, y, 1.0);
    y = fma(y, e, y);
    const double q = num * y;
    return fma(fma(-den, q, num), y, q);
}

// 2T F from the reduced energies x1 = e1/2T, x2 = e2/2T (the group kernel
// folds 1/2T into its row coefficients and its region Jacobian): with
// d = x1 - x2 = (e1 - e2)/2T,
//   near (|d| <= 1/16):  2T F = v1 v2 (2 sinhc d) / ((1+u1)(1+u2))
//   far:                 2T F = s [u2 - u1 | 1 - u1 u2] / ((1+u1)(1+u2) d)
// (the same branches and identities as bubble_F, one factor 2T throughout).
// v1 = exp(-|x1|).
__device__ __forceinline__ double bubble_F2T(double x1, double v1, double x2, const double* tab)
{
    const double d = x1 - x2;
    const double v2 = exp_neg(fabs(x2), tab);
    const double u1 = v1 * v1, u2 = v2 * v2;
    const double p = (1.0 + u1) * (1.0 + u2);
    const bool near = fabs(d) <= 0.0625;
    const bool neg1 = x1 < 0.0;
    const bool same = neg1 == (x2 < 0.0);
    double far = same ? (u2 - u1) : fma(-u1, u2, 1.0);
    far = neg1 ? -far : far;
    double num = far, den = p * d;
    // the near branch is needed only in the thin band |e(k) - e(k')| <= 2T/16
    // (all of the zone only near q = 0): a warp none of whose lanes is near
    // skips the series
    if (__any_sync(__activemask(), near)) {
        const double d2 = d * d;
        const double sinhc2 = fma(d2, fma(d2, fma(d2, fma(d2, 2.0 / 362880.0, 2.0 / 5040.0),
                                                   2.0 / 120.0), 2.0 / 6.0), 2.0);
        if (near) {
            num = (v1 * v2) * sinhc2;
            den = p;
        }
    }
    return div_nr(num, den);
}

// Omega derivative of the frequency integrals of the flow kinds (Sec. 2,
// regulator theta(k0) = k0^2 / (k0^2 + Omega^2), T = 0, measure dk0 / 2pi):
// the divided difference of Hdot(e) = e (3|e| + W) / (4 (|e| + W)^3) at
// (e1, e2) for ph and minus that at (e1, -e2) for pp.  With u = |e| + W:
// energies of one sign (Hdot odd and smooth there):
//   (-3 P^2 + 5 W S P - 2 W^2 (S^2 - P)) / (4 P^3),  P = u1 u2, S = u1 + u2
// (the exact divided difference of (3/u - 5W/u^2 + 2W^2/u^3) / 4);
// opposite signs (no cancellation):
//   (e1 (3|e1| + W) u2^3 - e2 (3|e2| + W) u1^3) / (4 u1^3 u2^3 (e1 - e2)).
__device__ __forceinline__ double flow_Fdot(double e1, double e2, double W, bool pp)
{
    if (pp) e2 = -e2;
    const double a1 = fabs(e1), a2 = fabs(e2);
    const double u1 = a1 + W, u2 = a2 + W;
    const double P = u1 * u2, S = u1 + u2;
    const bool same = (e1 >= 0.0) == (e2 >= 0.0);
    const double u13 = u1 * u1 * u1, u23 = u2 * u2 * u2;
    const double num_s = fma(-3.0 * P, P, W * fma(5.0 * S, P, -2.0 * W * fma(S, S, -P)));
    const double num_o = fma(e1 * fma(3.0, a1, W), u23, -e2 * fma(3.0, a2, W) * u13);
    const double num = same ? num_s : num_o;
    const double den = same ? 4.0 * P * P * P : 4.0 * u13 * u23 * (e1 - e2);
    const double D = div_nr(num, den);
    return pp ? -D : D;
}

// ---------------------------------------------------------------------------
// FP32-pipe evaluation of the shared-partition kernel (options.eval_fp32 with
// group_mode).  A float-float number is an unevaluated sum hi + lo of two FP32
// numbers (about 48 significant bits) on the FP32 pipe (64x the FP64 pipe on
// this GPU).  The building blocks are the published error-free
// transformations: Knuth's TwoSum, Dekker's FastTwoSum (|a| >= |b|) and the FMA
// form of TwoProduct, combined as in double-word arithmetic.
//
// Every thread carries two float-float numbers at a time, one per lane of a
// packed pair, through the two-wide FP32 instructions (add / mul / fma
// .rn.f32x2): they run at the pipe's full rate with half the issue slots of
// scalar code (measured: 62-63 packed instructions per clock and SM against
// 121-123 scalar ones), which leaves the slots for loads, table lookups and
// selects.  The scalar form of this kernel was bound by issue: 360 FP32
// instructions a node and half as many others kept the pipe at 0.58 of its
// rate.  Each lane is rounded as the scalar instruction rounds, so a lane's
// result does not depend on its partner.  A negated operand and one broadcast
// to both lanes are free (operand modifiers), so the code negates and
// broadcasts where the arithmetic wants it.
struct w2 {
    float2 hi, lo;
};

__device__ __forceinline__ f2 ff_from(double x)
{
    const float h = __double2float_rn(x);
    return {h, __double2float_rn(x - double(h))};
}
__device__ __forceinline__ float2 ff_st(f2 a) { return make_float2(a.hi, a.lo); }

__device__ __forceinline__ float2 dup(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __fadd2_rn(a, neg2(b)); }
// two scalar multiplications: the assembler may fuse a packed multiplication
// with the packed addition that takes its result (rounding modes notwithstanding),
// which would break the error-free transformations; __fmul_rn never fuses, and
// the pair costs the pipe what a packed one does
__device__ __forceinline__ float2 mul2(float2 a, float2 b)
{
    return make_float2(__fmul_rn(a.x, b.x), __fmul_rn(a.y, b.y));
}
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }

__device__ __forceinline__ w2 w_dup(float hi, float lo) { return {dup(hi), dup(lo)}; }
__device__ __forceinline__ w2 w_dup(float2 v) { return {dup(v.x), dup(v.y)}; }
// lane x from a, lane y from b (each a float-float number (hi, lo))
__device__ __forceinline__ w2 w_pair(float2 a, float2 b)
{
    return {make_float2(a.x, b.x), make_float2(a.y, b.y)};
}
__device__ __forceinline__ float2 w_x(w2 a) { return make_float2(a.hi.x, a.lo.x); }
__device__ __forceinline__ float2 w_y(w2 a) { return make_float2(a.hi.y, a.lo.y); }
__device__ __forceinline__ w2 w_zero() { return w_dup(0.0f, 0.0f); }
__device__ __forceinline__ w2 w_neg(w2 a) { return {neg2(a.hi), neg2(a.lo)}; }
// lane by lane: x from a or b by sx, y by sy
__device__ __forceinline__ w2 w_sel(bool sx, bool sy, w2 a, w2 b)
{
    return {make_float2(sx ? a.hi.x : b.hi.x, sy ? a.hi.y : b.hi.y),
            make_float2(sx ? a.lo.x : b.lo.x, sy ? a.lo.y : b.lo.y)};
}
__device__ __forceinline__ w2 w_two_sum(float2 a, float2 b)
{
    const float2 s = add2(a, b);
    const float2 bb = sub2(s, a);
    return {s, add2(sub2(a, sub2(s, bb)), sub2(b, bb))};
}
__device__ __forceinline__ w2 w_fast(float2 a, float2 b)   // |a| >= |b| (or a = 0)
{
    const float2 s = add2(a, b);
    return {s, sub2(b, sub2(s, a))};
}
__device__ __forceinline__ w2 w_add(w2 a, w2 b)
{
    const w2 s = w_two_sum(a.hi, b.hi);
    return w_fast(s.hi, add2(s.lo, add2(a.lo, b.lo)));
}
__device__ __forceinline__ w2 w_sub(w2 a, w2 b) { return w_add(a, w_neg(b)); }
// 1 + u for 0 <= u <= 1
__device__ __forceinline__ w2 w_one_plus(w2 u)
{
    const w2 s = w_fast(dup(1.0f), u.hi);
    return w_fast(s.hi, add2(s.lo, u.lo));
}
// the product's leading part p and its rounding error with the cross terms
__device__ __forceinline__ float2 w_prod_err(w2 a, w2 b, float2 p)
{
    float2 e = fma2(a.hi, b.hi, neg2(p));
    e = fma2(a.hi, b.lo, e);
    return fma2(a.lo, b.hi, e);
}
__device__ __forceinline__ w2 w_mul(w2 a, w2 b)
{
    const float2 p = mul2(a.hi, b.hi);
    return w_fast(p, w_prod_err(a, b, p));
}
// c a for an FP32 constant c
__device__ __forceinline__ w2 w_mul_f(float c, w2 a)
{
    const float2 p = mul2(dup(c), a.hi);
    const float2 e = fma2(dup(c), a.lo, fma2(dup(c), a.hi, neg2(p)));
    return w_fast(p, e);
}
// 2^k a: exact
__device__ __forceinline__ w2 w_scale(float c, w2 a) { return {mul2(dup(c), a.hi), mul2(dup(c), a.lo)}; }
__device__ __forceinline__ w2 w_sqr(w2 a)
{
    const float2 p = mul2(a.hi, a.hi);
    float2 e = fma2(a.hi, a.hi, neg2(p));
    e = fma2(add2(a.hi, a.hi), a.lo, e);
    return w_fast(p, e);
}
// a b + c, normalised
__device__ __forceinline__ w2 w_fma(w2 a, w2 b, w2 c)
{
    const float2 p = mul2(a.hi, b.hi);
    const float2 e = w_prod_err(a, b, p);
    const w2 s = w_two_sum(c.hi, p);
    return w_fast(s.hi, add2(s.lo, add2(e, c.lo)));
}
// c += a b with c an accumulator left unnormalised: hi takes the rounded
// running sum, lo every rounding error (exact TwoSum and TwoProduct errors and
// the cross terms), so lo stays within a few ulp of hi over a row of nodes;
// w_fast(hi, lo) normalises at the end.
__device__ __forceinline__ void w_acc(w2 a, w2 b, w2& c)
{
    const float2 p = mul2(a.hi, b.hi);
    const float2 e = w_prod_err(a, b, p);
    const w2 s = w_two_sum(c.hi, p);
    c.hi = s.hi;
    c.lo = add2(c.lo, add2(s.lo, e));
}
// a / b, b normal and non-zero: q1 = a_hi rcp(b_hi), one correction from the
// residual a - b q1 (its leading part a_hi - b_hi q1 is exact, Sterbenz).
__device__ __forceinline__ w2 w_div(w2 a, w2 b)
{
    const float2 r = make_float2(rcp_approx(b.hi.x), rcp_approx(b.hi.y));
    const float2 q1 = mul2(a.hi, r);
    const float2 p = mul2(b.hi, q1);
    const float2 e = fma2(b.hi, q1, neg2(p));
    float2 res = sub2(sub2(a.hi, p), e);
    res = fma2(neg2(b.lo), q1, res);
    res = add2(res, a.lo);
    return w_fast(q1, mul2(res, r));
}
// v, negated where `sign` has its sign bit set
__device__ __forceinline__ float flip_by(float v, float sign)
{
    return __int_as_float(__float_as_int(v) ^ (__float_as_int(sign) & int(0x80000000u)));
}
__device__ __forceinline__ w2 w_flip(w2 v, float2 sign)
{
    return {make_float2(flip_by(v.hi.x, sign.x), flip_by(v.hi.y, sign.y)),
            make_float2(flip_by(v.lo.x, sign.x), flip_by(v.lo.y, sign.y))};
}
__device__ __forceinline__ w2 w_abs(w2 a) { return w_flip(a, a.hi); }

// exp(-a) for a float-float a >= 0 (Tang's table-driven method, as exp_neg):
// a = k ln2/64 + r, k = rint(64 a / ln2), e^-a = 2^(-k/64) e^-r.  ln2/64 is
// split as C1 + C2 + C3 with C1 of 9 significant bits, so k C1 is exact for
// k < 2^15 and a_hi - k C1 is exact (Sterbenz); r is then formed in
// float-float.  Its first sum is a FastTwoSum: a_hi - k C1 is a multiple of
// ulp(a_hi) (C1 is a multiple of 2^-15 and a_hi < 50), so it is zero or at
// least |a_lo|.  e^t (t = -r, |t| <= 0.0055) = 1 + t + t^2/2 + t^3 (1/6 + t/24
// + t^2/120): the first three terms in float-float, the rest (< 3e-8) in FP32
// (error < 4e-15); truncation t^6/720 < 4e-17.  2^(j/64) comes from a
// float-float table and 2^m (m >= -73) scales both parts exactly.  a >= 50
// gives 0 (e^-50 < 2e-22: the kernel F only uses v^2 and products of v there,
// which flush to zero in FP32); a pair with both lanes there returns at once.
__device__ __forceinline__ w2 w_exp_neg(w2 a, const float2* tab)
{
    const bool zx = a.hi.x >= 50.0f, zy = a.hi.y >= 50.0f;
    if (zx && zy) return w_zero();
    const float C1 = 0.010833740234375f;          // 0x1.63p-7
    const float C2 = -3.3155381515825866e-06f;
    const float C3 = 2.572804640231345e-14f;
    // k = rint(64 a_hi / ln2) by the shift 1.5 * 2^23: the sum lies in
    // [2^23, 2^24), where the float grid is the integers, so its low encoding
    // bits are k (two FP32-pipe instructions in place of a float rounding and
    // a float-to-integer conversion)
    const float2 kt = fma2(a.hi, dup(92.33248138427734f), dup(12582912.0f));
    const float2 k = sub2(kt, dup(12582912.0f));
    const float2 t1 = fma2(neg2(k), dup(C1), a.hi);          // exact
    const w2 s1 = w_fast(t1, a.lo);
    const float2 p2 = mul2(k, dup(C2));
    const float2 e2 = fma2(k, dup(C2), neg2(p2));
    const w2 s2 = w_two_sum(s1.hi, neg2(p2));
    float2 lo = add2(s2.lo, s1.lo);
    lo = sub2(lo, e2);
    lo = fma2(neg2(k), dup(C3), lo);
    const w2 r = w_fast(s2.hi, lo);
    const float2 th = neg2(r.hi), tl = neg2(r.lo);           // t = -r
    const float2 h = mul2(th, th);
    const float2 hl = fma2(th, th, neg2(h));                 // th^2 = h + hl
    float2 q = fma2(th, dup(1.0f / 120.0f), dup(1.0f / 24.0f));
    q = fma2(th, q, dup(1.0f / 6.0f));
    const float2 c = mul2(mul2(h, th), q);
    const w2 S = w_fast(th, mul2(dup(0.5f), h));             // t + t^2/2, leading parts
    float2 sl = add2(S.lo, tl);
    sl = fma2(dup(0.5f), hl, sl);
    sl = fma2(th, tl, sl);
    sl = add2(sl, c);
    const w2 P0 = w_fast(dup(1.0f), S.hi);
    const w2 P = w_fast(P0.hi, add2(P0.lo, sl));
    const int nx = 0x4B400000 - __float_as_int(kt.x);        // -k
    const int ny = 0x4B400000 - __float_as_int(kt.y);
    // 2^(j/64), j = -k mod 64; 2^m, m = floor(-k / 64)
    const w2 y = w_mul(P, w_pair(tab[nx & 63], tab[ny & 63]));
    const float2 sc = make_float2(__int_as_float(((nx >> 6) + 127) << 23),
                                  __int_as_float(((ny >> 6) + 127) << 23));
    const w2 v = {mul2(y.hi, sc), mul2(y.lo, sc)};
    return w_sel(zx, zy, w_zero(), v);
}

// 2T F(x1, x2) in float-float from the reduced energies (x = e/2T, the same
// branches and identities as bubble_F2T): d = x1 - x2,
//   near (|d| <= 1/16):  v1 v2 (2 sinhc d) / ((1+u1)(1+u2))
//   far:                 s [u2 - u1 | 1 - u1 u2] / ((1+u1)(1+u2) d)
// 2 sinhc d = 2 + d^2/3 + d^4/60 + d^6/2520 + d^8/181440 (next term < 5e-20
// at |d| = 1/16), the d^2/3 term in float-float.  v1 = exp(-|x1|).
__device__ __forceinline__ w2 w_bubble_F2T(w2 x1, w2 v1, w2 x2, const float2* tab)
{
    const w2 d = w_sub(x1, x2);
    const w2 v2 = w_exp_neg(w_abs(x2), tab);
    const w2 u1 = w_sqr(v1), u2 = w_sqr(v2);
    const w2 p = w_mul(w_one_plus(u1), w_one_plus(u2));
    const bool sx = (__float_as_int(x1.hi.x) ^ __float_as_int(x2.hi.x)) >= 0;   // same sign
    const bool sy = (__float_as_int(x1.hi.y) ^ __float_as_int(x2.hi.y)) >= 0;
    const w2 u12 = w_mul(u1, u2);
    w2 num = w_sub(w_sel(sx, sy, u2, w_dup(1.0f, 0.0f)), w_sel(sx, sy, u1, u12));
    num = w_flip(num, x1.hi);
    w2 den = w_mul(p, d);
    const bool nearx = fabsf(d.hi.x) <= 0.0625f, neary = fabsf(d.hi.y) <= 0.0625f;
    if (__any_sync(__activemask(), nearx || neary)) {
        const w2 d2 = w_sqr(d);
        const float2 g = d2.hi;
        const float2 tail = mul2(mul2(g, g), fma2(g, fma2(g, dup(1.0f / 181440.0f), dup(1.0f / 2520.0f)),
                                                  dup(1.0f / 60.0f)));
        const w2 third = w_mul(d2, w_dup(0.3333333432674408f, -9.934107758624577e-09f));
        const w2 S0 = w_fast(dup(2.0f), third.hi);    // 2 > d^2/3: exact
        const w2 S = w_fast(S0.hi, add2(S0.lo, add2(third.lo, tail)));
        num = w_sel(nearx, neary, w_mul(w_mul(v1, v2), S), num);
        den = w_sel(nearx, neary, p, den);
    }
    return w_div(num, den);
}

// Omega derivative of the flow kinds' frequency integrals in float-float (the
// same formulas as flow_Fdot's ph case; e1, e2 energies, W = Omega as
// float-float).  Either form runs only in warps that hold such a node.
__device__ __forceinline__ w2 w_flow_Fdot(w2 e1, w2 e2, w2 W)
{
    const w2 a1 = w_abs(e1), a2 = w_abs(e2);
    const w2 u1 = w_add(a1, W), u2 = w_add(a2, W);
    const bool sx = (e1.hi.x < 0.0f) == (e2.hi.x < 0.0f);
    const bool sy = (e1.hi.y < 0.0f) == (e2.hi.y < 0.0f);
    w2 num = w_zero(), den = w_dup(1.0f, 0.0f);
    const unsigned act = __activemask();
    if (__any_sync(act, sx || sy)) {
        // -3 P^2 + W (5 S P - 2 W (S^2 - P))
        const w2 P = w_mul(u1, u2), S = w_add(u1, u2);
        const w2 inner = w_sub(w_mul(w_mul_f(5.0f, S), P),
                               w_mul(w_scale(2.0f, W), w_sub(w_sqr(S), P)));
        const w2 PP = w_sqr(P);
        num = w_sub(w_mul(W, inner), w_mul_f(3.0f, PP));
        den = w_scale(4.0f, w_mul(P, PP));
    }
    if (__any_sync(act, !sx || !sy)) {
        const w2 u13 = w_mul(u1, w_sqr(u1)), u23 = w_mul(u2, w_sqr(u2));
        const w2 g1 = w_mul(e1, w_add(w_mul_f(3.0f, a1), W));
        const w2 g2 = w_mul(e2, w_add(w_mul_f(3.0f, a2), W));
        const w2 no = w_sub(w_mul(g1, u23), w_mul(g2, u13));
        const w2 dd = w_mul(w_scale(4.0f, w_mul(u13, u23)), w_sub(e1, e2));
        num = w_sel(sx, sy, num, no);
        den = w_sel(sx, sy, den, dd);
    }
    return w_div(num, den);
}

// Diagnostics for paid_check_math: which = 0: exp_neg(x), 1: div_nr(x, y),
// 2: w_exp_neg(x) (x rounded to float-float), 3: w_bubble_F2T(x, y),
// 4: bubble_F2T(x, y) (FP64), 5: w_flow_Fdot(x, y) with Omega = 0.1 (ph),
// 6: flow_Fdot(x, y) with Omega = 0.1 (ph).  The packed functions take elements
// i and i xor 1 as their two lanes, element i in lane i & 1.
__global__ void k_check_math(int which, int64_t n, const double* x, const double* y, double* out)
{
    __shared__ double tab[64];
    __shared__ float2 tabf[64];
    if (threadIdx.x < 64) {
        tab[threadIdx.x] = c_exp2d[threadIdx.x];
        const f2 a = ff_from(c_exp2d[threadIdx.x]);
        tabf[threadIdx.x] = make_float2(a.hi, a.lo);
    }
    __syncthreads();
    const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    if (i >= n) return;
    auto pair = [&](const double* a) {
        const int64_t i0 = i & ~int64_t(1), i1 = i0 + 1 < n ? i0 + 1 : i0;
        return w_pair(ff_st(ff_from(a[i0])), ff_st(ff_from(a[i1])));
    };
    auto put = [&](w2 r) {
        const float2 v = (i & 1) ? w_y(r) : w_x(r);
        out[i] = double(v.x) + double(v.y);
    };
    switch (which) {
    case 0: out[i] = exp_neg(x[i], tab); break;
    case 1: out[i] = div_nr(x[i], y[i]); break;
    case 2: put(w_exp_neg(pair(x), tabf)); break;
    case 3: put(w_bubble_F2T(pair(x), w_exp_neg(w_abs(pair(x)), tabf), pair(y), tabf)); break;
    case 4: out[i] = bubble_F2T(x[i], exp_neg(fabs(x[i]), tab), y[i], tab); break;
    case 5: put(w_flow_Fdot(pair(x), pair(y), w_dup(ff_st(ff_from(0.1))))); break;
    default: out[i] = flow_Fdot(x[i], y[i], 0.1, false); break;
    }
}

cudaError_t launch_check_math(int which, int64_t n, const double* x, const double* y, double* out,
                              cudaStream_t s)
{
    if (n <= 0) return cudaSuccess;
    k_check_math<<<int((n + 255) / 256), 256, 0, s>>>(which, n, x, y, out);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Shared-partition (group) evaluation: one region of a (kind, q) group gives
// Q_N and Q_2N of every (l, m) pair of the group's batch at once.  With
// g = (1, cos, sin) every form factor is f_n(k) = sum C_n[a][b] g_a(kx) g_b(ky),
// so with k' = k + q (ph) or q - k (pp)
//   f_l(k) f_m(k') = sum C_l[a][b] C_m[c][d] X_ac(kx) Y_bd(ky),
//   X_ac = g_a(kx) g_c(kx'),   Y_bd = g_b(ky) g_d(ky'),
// and the rule applied to every pair needs only the 81 moments
//   M[ac][bd] = sum_i wx_i X_ac(x_i) R_i[bd],   R_i[bd] = sum_j wy_j F_ij Y_bd(y_j)
// and their coarse-rule counterparts: the kernel F once per node, 81 NF FMA
// (fine) + 81 (N+1) (coarse) for the moments, at most 4 terms per pair.
// Block: NF = 2N+1 threads per region (thread i owns fine row i, and column
// i for the shared column data, and moment cells i, i + NF, ...),
// GroupShape<N>::R regions per block.
template <int N> struct GroupShape;
template <> struct GroupShape<4> { static constexpr int R = 14; };   // 126 threads
template <> struct GroupShape<6> { static constexpr int R = 9; };    // 117 threads
template <> struct GroupShape<8> { static constexpr int R = 7; };    // 119 threads
template <> struct GroupShape<10> { static constexpr int R = 6; };   // 126 threads
template <> struct GroupShape<12> { static constexpr int R = 5; };   // 125 threads

constexpr int64_t kNodesMax = 6000;   // regions of a round (the FP32-pipe kernel's nodes split)

// The first energy's half of the kernel F, shared between groups.  x1 = e(k)/2T and
// exp(-|x1|) at a region's nodes depend on T and the region only, not on q or on ph /
// pp, and a call's groups meet the same regions (a flow step's 641,744 evaluations at
// T = 0.05 are of some thousand regions): 65 of a node's 290 FP32 instructions.  In a
// round of the rows split, one pass finds the distinct (T, region) entries, a second
// evaluates both numbers once for each, and the evaluation reads its 32 bytes per row
// pair and column (10 KB a region, mostly from L2) where it would compute them.  A
// block holds x1 and then exp(-|x1|), column by column with the row pairs side by side,
// so that a warp's 16-byte loads are contiguous.  Measured, evaluation of the flow step
// with these passes: 4.68 ms against 5.34 without; row pair by row pair 4.76 (a warp's
// loads in 32 lines); with u1 and 1 + u1 in the table as well 4.70.  T = 0.01 on 12 x 12,
// where the tables leave L2: 13.9 against 14.8.  The FP64 kernel reads FP64 tables (12
// of a node's 63 FP64 instructions): 288 groups at T = 0.05 17.0 -> 14.7 ms a call.
//
// A table is worth its block only where enough regions read it, so once the distinct
// entries are counted the round decides: the tables are built and read when they have
// room for every distinct entry and these repeat often enough (first_quarters).  The
// group count alone, which decided before, cost calls with few momenta at each of many
// temperatures: 2,048 temperatures from 0.1 on, one momentum each, FP32 pipe, N = 12 27.1
// ms against 24.2, N = 8 28.2 against 25.3; 512 temperatures, N = 4 14.4 against 12.0.
//
// The tables live in the pool buffers that the round's split has not written yet:
// hash slots in err[next], per entry its distinct index (its table block) or the entry
// that holds it in own[next], per distinct index an entry in key[next], the blocks in
// vval[next] and verr[next].
struct First {
    uint32_t* slot;            // hash table: entry + 1, or 0
    uint64_t mask;             // its size - 1 (a power of two)
    uint32_t* uid;             // per entry: distinct index, kShareRef | entry, or kNoShare
    uint32_t* rep;             // per distinct index: an entry
    float4 *b0, *b1;           // blocks [2][column][row pair] (b1 after nb0 of them)
    uint32_t nb0, room;
    int block;                 // float4 per block
};

__device__ __forceinline__ bool first_sharing(const Work& w, int64_t n)
{
    return w.share && n > kNodesMax && n < kShareMax;
}
template <int N>
__device__ __forceinline__ First first_view(const Work& w)
{
    const int nxt = w.ls->cur ^ 1;
    const int64_t n = w.ls->n_eval;
    First f;
    f.block = 2 * (N + 1) * (2 * N + 1);
    uint64_t size = 1;
    while (size < uint64_t(2 * n)) size <<= 1;
    while (size > uint64_t(2 * w.cap)) size >>= 1;
    f.slot = reinterpret_cast<uint32_t*>(w.err[nxt]);
    f.mask = size - 1;
    f.uid = w.own[nxt];
    f.rep = reinterpret_cast<uint32_t*>(w.key[nxt]);
    f.b0 = reinterpret_cast<float4*>(w.vval[nxt]);
    f.b1 = reinterpret_cast<float4*>(w.verr[nxt]);
    const int64_t bytes = 16 * int64_t(f.block);
    f.nb0 = uint32_t(min(w.cap * 8 * kGroupPairs / bytes, kShareMax / 2));
    f.room = f.nb0 + uint32_t(min(w.cap * 4 * kGroupPairs / bytes, kShareMax / 2));
    return f;
}
__device__ __forceinline__ float4* first_block(const First& f, uint32_t b)
{
    return b < f.nb0 ? f.b0 + size_t(b) * f.block : f.b1 + size_t(b - f.nb0) * f.block;
}
// after k_first_insert: whether this round builds and reads the tables
template <int N, bool FP32>
__device__ __forceinline__ bool first_used(const RoundCounts& r, const First& f)
{
    constexpr unsigned long long q = first_quarters(N, FP32);
    return q > 0 && r.distinct <= f.room && q * r.distinct <= 4 * r.sharable;
}
// the table of entry t's region (first_used), or null
__device__ __forceinline__ const float4* first_find(const First& f, int64_t t)
{
    uint32_t u = f.uid[t];
    if (u == kNoShare) return nullptr;
    if (u & kShareRef) u = f.uid[u & ~kShareRef];
    return first_block(f, u);
}

template <int N>
__global__ void k_first_clear(Work w)
{
    if (!first_sharing(w, w.ls->n_eval)) return;
    const First f = first_view<N>(w);
    const uint64_t stride = uint64_t(gridDim.x) * blockDim.x;
    const uint64_t i0 = uint64_t(blockIdx.x) * blockDim.x + threadIdx.x;
    for (uint64_t i = i0; i <= f.mask; i += stride) f.slot[i] = 0u;
    if (i0 == 0) w.totals->unsharable = w.totals->distinct = w.totals->unshared = 0ull;
}

// (six blocks per SM: at eight, 32 registers, the loop spills)
constexpr int kInsertBlocks = 6;
template <int N>
__global__ void __launch_bounds__(256, kInsertBlocks) k_first_insert(Work w)
{
    if (!first_sharing(w, w.ls->n_eval)) return;
    const First f = first_view<N>(w);
    const int cur = w.ls->cur;
    const int64_t n = w.ls->n_eval;
    const int lane = threadIdx.x & 31;
    const int64_t stride = int64_t(gridDim.x) * blockDim.x;
    unsigned left_out = 0;
    for (int64_t t0 = int64_t(blockIdx.x) * blockDim.x + threadIdx.x - lane; t0 < n; t0 += stride) {
        const int64_t t = t0 + lane;
        uint32_t u = kNoShare;
        bool mine = false;
        if (t < n) {
            const uint2 e = w.evl[t];
            const uint32_t mt = w.meta[e.y];
            if (meta_kind(mt) != PH && meta_kind(mt) != PP) {
                ++left_out;
            } else {
                const uint64_t key = w.key[cur][e.x];
                const double h2 = w.batches[meta_batch(mt)].inv2T;
                uint64_t h = key ^ (uint64_t(__double_as_longlong(h2)) * 0x9e3779b97f4a7c15ull);
                h = (h ^ (h >> 30)) * 0xbf58476d1ce4e5b9ull;   // splitmix64's finaliser
                h = (h ^ (h >> 27)) * 0x94d049bb133111ebull;
                h ^= h >> 31;
                for (int p = 0; p < kShareProbes; ++p) {
                    uint32_t* slot = &f.slot[(h + p) & f.mask];
                    uint32_t old = __ldcg(slot);   // most regions are there already
                    if (old == 0u) old = atomicCAS(slot, 0u, uint32_t(t) + 1u);
                    if (old == 0u) { mine = true; break; }
                    const uint2 o = w.evl[old - 1u];
                    if (w.key[cur][o.x] == key &&
                        w.batches[meta_batch(w.meta[o.y])].inv2T == h2) {
                        u = kShareRef | (old - 1u);
                        break;
                    }
                }
                if (!mine && u == kNoShare) left_out += 0x10000u;   // its probes ran out
            }
        }
        const unsigned m = __ballot_sync(0xffffffffu, mine);
        unsigned long long base = 0;
        if (lane == 0 && m) base = atomicAdd(&w.totals->distinct, (unsigned long long)__popc(m));
        base = __shfl_sync(0xffffffffu, base, 0);
        if (mine) {
            u = uint32_t(base) + uint32_t(__popc(m & ((1u << lane) - 1u)));
            f.rep[u] = uint32_t(t);
        }
        if (t < n) f.uid[t] = u;
    }
    add_left_out(w, left_out);
}

template <int N>
struct GroupSmem {
    static constexpr int NF = 2 * N + 1, R = GroupShape<N>::R;
    double X[R][NF][9];      // X_ac at the fine rows
    double Y[R][NF][9];      // Y_bd at the fine columns
    double CY[R][NF][2];     // cos ky, cos ky' at the fine columns
    double Rf[R][NF][9];     // fine row sums R_i[bd]
    double Rc[R][N + 1][9];  // coarse row sums (even rows)
    double Mf[R][9][9];      // fine moments
    double Mc[R][9][9];      // coarse moments
    double C[R][4];          // sin, cos of the region centre (x, y) times pi
    double tab[64];          // 2^(j/64)
};

// the FP64 kernel's table blocks, x1 then exp(-|x1|) as [column][row]: NF threads per
// region, thread i owning row i and column i
template <int N>
__global__ void __launch_bounds__(GroupShape<N>::R * (2 * N + 1)) k_first_eval_fp64(Work w, Lattice lat)
{
    constexpr int NF = 2 * N + 1, R = GroupShape<N>::R;
    static_assert(2 * NF * NF * 8 <= 2 * (N + 1) * NF * 16, "fits a block");
    __shared__ double C[R][4], cys[R][NF], tab[64];
    const RoundCounts rc = round_counts(w);
    if (!first_sharing(w, rc.n)) return;
    const First f = first_view<N>(w);
    const bool used = first_used<N, false>(rc, f);
    note_sharing(w, rc, used, f.room);
    if (!used) return;
    const int cur = w.ls->cur, v = rule_variant(N);
    const uint32_t count = uint32_t(rc.distinct);
    const int rho = threadIdx.x / NF, i = threadIdx.x % NF;
    if (threadIdx.x < 64) tab[threadIdx.x] = c_exp2d[threadIdx.x];
    const double tA = -2.0 * lat.t, tB = -4.0 * lat.tp;
    for (uint32_t u0 = blockIdx.x * R; u0 < count; u0 += gridDim.x * R) {
        const uint32_t u = u0 + rho;
        const bool live = u < count;
        uint32_t L = 0, g = 0;
        if (live) {
            const uint2 e = w.evl[f.rep[u]];
            g = e.y;
            const uint64_t key = w.key[cur][e.x];
            L = key_level(key);
            if (i < 2) {
                const uint32_t ic = i == 0 ? key_ix(key) : key_iy(key);
                sincospi(fma(double(2 * ic + 1), ldexp(1.0, -int(L)), -1.0), &C[rho][2 * i],
                         &C[rho][2 * i + 1]);
            }
        }
        __syncthreads();
        double A1 = 0.0, B1 = 0.0;
        if (live) {
            const double sxc = C[rho][0], cxc = C[rho][1], syc = C[rho][2], cyc = C[rho][3];
            const int ii = i <= N ? i : 2 * N - i;
            const double co = c_co[v][L][ii];
            const double so = i <= N ? c_so[v][L][ii] : -c_so[v][L][ii];
            const double cx = fma(cxc, co, -sxc * so);
            cys[rho][i] = fma(cyc, co, -syc * so);
            const double h1 = w.batches[meta_batch(w.meta[g])].inv2T;
            A1 = fma(tA, cx, -lat.mu) * h1;
            B1 = fma(tB, cx, tA) * h1;
        }
        __syncthreads();
        if (live) {
            double* out = reinterpret_cast<double*>(first_block(f, u)) + i;
#pragma unroll 1
            for (int j = 0; j < NF; ++j) {
                const double x1 = fma(B1, cys[rho][j], A1);
                out[j * NF] = x1;
                out[(NF + j) * NF] = exp_neg(fabs(x1), tab);
            }
        }
        __syncthreads();
    }
}

template <int N>
__global__ void __launch_bounds__(GroupShape<N>::R * (2 * N + 1))
k_eval_group(Work w, Lattice lat, double* rule_q2, double* rule_d)
{
    constexpr int NF = 2 * N + 1, R = GroupShape<N>::R;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    GroupSmem<N>& S = *reinterpret_cast<GroupSmem<N>*>(smem_raw);
    const int v = rule_variant(N);
    const int cur = w.ls->cur;
    const int64_t n_eval = w.ls->n_eval;
    const int rho = threadIdx.x / NF, i = threadIdx.x % NF;
    const double tA = -2.0 * lat.t, tB = -4.0 * lat.tp;
    if (threadIdx.x < 64) S.tab[threadIdx.x] = c_exp2d[threadIdx.x];
    const RoundCounts rc = round_counts(w);
    const First fs = first_sharing(w, rc.n) ? first_view<N>(w) : First{};
    const bool first = first_sharing(w, rc.n) && first_used<N, false>(rc, fs);
    for (int64_t chunk = blockIdx.x; chunk * R < n_eval; chunk += gridDim.x) {
        const int64_t t = chunk * R + rho;
        const bool live = t < n_eval;
        uint32_t pos = 0, g = 0, L = 0;
        int kind = PH, P = 0;
        const DevBatch* B = nullptr;
        const double* known = nullptr;   // x1 and exp(-|x1|) of this region's row i
        double A1 = 0.0, B1 = 0.0, A2 = 0.0, B2 = 0.0;
        uint64_t key = 0;
        if (live) {
            if (first) {
                const float4* f = first_find(fs, t);
                known = f ? reinterpret_cast<const double*>(f) + i : nullptr;
            }
            const uint2 e = w.evl[t];
            pos = e.x;
            g = e.y;
            key = w.key[cur][pos];
            L = key_level(key);
            if (i < 2) {   // the exact dyadic centre / pi: -1 + (2 ix + 1) 2^-L, x then y
                const uint32_t ic = i == 0 ? key_ix(key) : key_iy(key);
                sincospi(fma(double(2 * ic + 1), ldexp(1.0, -int(L)), -1.0), &S.C[rho][2 * i],
                         &S.C[rho][2 * i + 1]);
            }
        }
        __syncthreads();
        if (live) {
            const uint32_t mt = w.meta[g];
            B = &w.batches[meta_batch(mt)];
            kind = meta_kind(mt);
            P = B->npairs;
            const QTrig tq = w.trig[g];     // flow kinds: rotation by q/2
            const bool pp = kind == PP, flow = is_flow(kind);
            const double sxc = S.C[rho][0], cxc = S.C[rho][1];
            const double syc = S.C[rho][2], cyc = S.C[rho][3];
            const int ii = i <= N ? i : 2 * N - i;
            const double co = c_co[v][L][ii];
            const double so = i <= N ? c_so[v][L][ii] : -c_so[v][L][ii];
            // row i (x) and column i (y) of the fine grid, and the shifted k'
            const double cx = fma(cxc, co, -sxc * so), sx = fma(sxc, co, cxc * so);
            const double cy = fma(cyc, co, -syc * so), sy = fma(syc, co, cyc * so);
            const double cx2 = pp ? fma(tq.cqx, cx, tq.sqx * sx) : fma(cx, tq.cqx, -sx * tq.sqx);
            const double sx2 = pp ? fma(tq.sqx, cx, -tq.cqx * sx) : fma(sx, tq.cqx, cx * tq.sqx);
            const double cy2 = pp ? fma(tq.cqy, cy, tq.sqy * sy) : fma(cy, tq.cqy, -sy * tq.sqy);
            const double sy2 = pp ? fma(tq.sqy, cy, -tq.cqy * sy) : fma(sy, tq.cqy, cy * tq.sqy);
            // flow kinds: both form factors at k (symmetric routing)
            const double gx[3] = {1.0, cx, sx};
            const double gx2[3] = {1.0, flow ? cx : cx2, flow ? sx : sx2};
            const double gy[3] = {1.0, cy, sy};
            const double gy2[3] = {1.0, flow ? cy : cy2, flow ? sy : sy2};
#pragma unroll
            for (int a = 0; a < 3; ++a)
#pragma unroll
                for (int c = 0; c < 3; ++c) {
                    S.X[rho][i][3 * a + c] = gx[a] * gx2[c];
                    S.Y[rho][i][3 * a + c] = gy[a] * gy2[c];
                }
            if (flow) {
                // e(k + q/2) and e(k - q/2): cos(k +- q/2) = cos k cos q/2 -+ sin k sin q/2
                const double cxp = fma(cx, tq.cqx, -sx * tq.sqx), cxm = fma(cx, tq.cqx, sx * tq.sqx);
                S.CY[rho][i][0] = fma(cy, tq.cqy, -sy * tq.sqy);
                S.CY[rho][i][1] = fma(cy, tq.cqy, sy * tq.sqy);
                A1 = fma(tA, cxp, -lat.mu);
                B1 = fma(tB, cxp, tA);
                A2 = fma(tA, cxm, -lat.mu);
                B2 = fma(tB, cxm, tA);
            } else {
                S.CY[rho][i][0] = cy;
                S.CY[rho][i][1] = cy2;
                // x = e / 2T = A + B cos ky along row i, for k and for k' (for pp
                // the second energy enters with its sign flipped)
                const double h1 = B->inv2T, h2 = pp ? -B->inv2T : B->inv2T;
                A1 = fma(tA, cx, -lat.mu) * h1;
                B1 = fma(tB, cx, tA) * h1;
                A2 = fma(tA, cx2, -lat.mu) * h2;
                B2 = fma(tB, cx2, tA) * h2;
            }
        }
        const bool every = __syncthreads_and(!live || known);
        if (live) {
            double rf[9], rc[9];
#pragma unroll
            for (int k = 0; k < 9; ++k) { rf[k] = 0.0; rc[k] = 0.0; }
            auto sums = [&](int j, double F) {
                const double wf = c_wf[v][j] * F;
#pragma unroll
                for (int k = 0; k < 9; ++k) rf[k] = fma(wf, S.Y[rho][j][k], rf[k]);
                if ((j & 1) == 0) {
                    const double wc = c_wc[v][j >> 1] * F;
#pragma unroll
                    for (int k = 0; k < 9; ++k) rc[k] = fma(wc, S.Y[rho][j][k], rc[k]);
                }
            };
            if (every) {
                // the whole block's first energies are in the tables
#pragma unroll 2
                for (int j = 0; j < NF; ++j) {
                    const double x1 = __ldg(known + j * NF), v1 = __ldg(known + (NF + j) * NF);
                    sums(j, bubble_F2T(x1, v1, fma(B2, S.CY[rho][j][1], A2), S.tab));
                }
            } else {
#pragma unroll
                for (int j = 0; j < NF; ++j) {
                    // OVERLAP: 1; bubbles: 2T F (1/2T is in the Jacobian); flow: dF/dOmega
                    double F = 1.0;
                    const double x1 = fma(B1, S.CY[rho][j][0], A1);
                    const double x2 = fma(B2, S.CY[rho][j][1], A2);
                    if (is_flow(kind))
                        F = flow_Fdot(x1, x2, B->T, kind == FLOW_PP);
                    else if (kind != OVERLAP)
                        F = bubble_F2T(x1, exp_neg(fabs(x1), S.tab), x2, S.tab);
                    sums(j, F);
                }
            }
            // the row's own rule weight (fine, and coarse on the even rows)
            // goes into its sums, so the moments below are plain dot products
            const double wr = c_wf[v][i];
#pragma unroll
            for (int k = 0; k < 9; ++k) S.Rf[rho][i][k] = wr * rf[k];
            if ((i & 1) == 0) {
                const double wrc = c_wc[v][i >> 1];
#pragma unroll
                for (int k = 0; k < 9; ++k) S.Rc[rho][i >> 1][k] = wrc * rc[k];
            }
        }
        __syncthreads();
        if (live) {
            // moments M[ac][bd]: the 81 (ac, bd) cells dealt over the region's
            // NF threads (all of them busy, rather than one thread per ac)
            for (int u = i; u < 81; u += NF) {
                const int ac = u / 9, bd = u - 9 * (u / 9);
                double mf = 0.0, mc = 0.0;
#pragma unroll
                for (int r = 0; r < NF; ++r) mf = fma(S.X[rho][r][ac], S.Rf[rho][r][bd], mf);
#pragma unroll
                for (int r = 0; r <= N; ++r) mc = fma(S.X[rho][2 * r][ac], S.Rc[rho][r][bd], mc);
                S.Mf[rho][ac][bd] = mf;
                S.Mc[rho][ac][bd] = mc;
            }
        }
        __syncthreads();
        if (live) {
            const double scale =
                ldexp(0.25, -2 * int(L)) * (kind == PH || kind == PP ? B->inv2T : 1.0);
            for (int p = i; p < P; p += NF) {
                const int l = B->lm[2 * p], m = B->lm[2 * p + 1];
                double q2 = 0.0, q1 = 0.0;
                if (l >= 0 && m >= 0 && l < w.nff && m < w.nff) {
                    for (int k1 = 0; k1 < c_ffn[l]; ++k1)
                        for (int k2 = 0; k2 < c_ffn[m]; ++k2) {
                            const double c = c_ffc[l][k1] * c_ffc[m][k2];
                            const int ac = 3 * c_ffa[l][k1] + c_ffa[m][k2];
                            const int bd = 3 * c_ffb[l][k1] + c_ffb[m][k2];
                            q2 = fma(c, S.Mf[rho][ac][bd], q2);
                            q1 = fma(c, S.Mc[rho][ac][bd], q1);
                        }
                }
                q2 *= scale;
                q1 *= scale;
                if (rule_q2) {
                    rule_q2[t * P + p] = q2;
                    rule_d[t * P + p] = q1 - q2;
                } else {
                    const size_t o = size_t(pos) * size_t(w.vstride) + size_t(p);
                    w.vval[cur][o] = q2;
                    w.verr[cur][o] = float(fabs(q1 - q2));
                }
            }
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------------------
// The FP32-pipe form of the shared-partition kernel (options.eval_fp32 with
// group_mode).  Same rule and data flow as k_eval_group, with every per-node,
// per-row and per-region quantity an unevaluated pair of FP32 numbers on the
// FP32 pipe: the node abscissae (rotations of the region centre), the reduced
// energies, the kernel F, the row sums, the moments, the pair combinations and
// the Jacobian.  FP64 remains for the two sincospi of the exact dyadic centre,
// the conversions of the per-region inputs, and each pair value's final
// conversion to FP64.
//
// The moments are taken in the Fourier basis phi = (1, cos k, sin k, cos 2k,
// sin 2k) of each direction instead of the nine products X_ac = g_a(k) g'_c(k')
// (g = (1, cos k, sin k) at k, g' the same at k' = k + q, or q - k for pp, or
// k for the flow kinds): every product is a fixed combination of the five
// (cos k cos k' = cos q (1 + cos 2k) / 2 - s sin q sin 2k / 2, ...), so a row
// needs 5 sums instead of 9 and a region 25 moments instead of 81, and the 81
// product moments follow from two small exact transforms per rule
// (w_fourier_to_products).
//
// What bounds it, and the two splits.  The FP32 pipe's operand reads are the
// limit: with three distinct registers a packed FMA issues at 0.6 of the pipe's
// rate and an addition at 0.9 (two reads a clock and scheduler; independent
// chains in registers, 20 warps per SM: a float-float accumulation takes 8.2
// clocks per SM and packed warp where its 12 instructions would take 6.0, a
// product 5.6 for 3.5), so about 0.7 of the nominal rate is what this mix
// reaches.  Every region's arithmetic is the same in both splits, operation by
// operation, so a region's results depend on neither the split nor its place.
//
// Rows (many regions): a thread owns an even and the next odd fine row of one
// region, one per packed lane: N+1 threads a region, the last with one row.
// The coarse rule wants the even row only: its five column sums run two to a
// pair with that lane's F in both lanes (three accumulations instead of five).
// R regions per block so that the last warp is nearly full (N = 12: 156 of 160
// lanes), B resident blocks for 20 warps per SM (96 registers).  Measured on
// the 93,312-integral flow step (641,744 regions from start level 3, evaluation per step): 12
// regions x 4 blocks 5.35 ms, x 3 5.97, x 5 (72 registers, spills) 5.69, 17 x 3
// 5.46, 9 x 5 5.41, 7 x 7 5.68; scalar code, one row per thread, 6.12.
//
// Nodes (few regions): one task per column of a row pair for F, kept in shared
// memory, then one per row pair and basis function for the row sums, so that a
// block is through with its regions after some 10 us instead of 40: 240 regions
// in three rounds 48 us instead of 127 (scalar rows: 88), 3,024 in six rounds
// 110 us instead of 216 (155).  Up to Rn regions per block, fewer when there are
// not enough for every block of the grid.  On many regions it is slower (the flow
// step: 6.2 ms): F goes through shared memory.  kNodesMax is where the two meet,
// measured at 3,000 / 6,000 / 10,000: 15,296 regions in six rounds 274 / 242 / 258
// us, 38,448 in six 445 / 447 / 478 us.  In one launch the two splits meet near 5,500
// regions at N = 4 and 6, 6,500 (flow kinds 9,500) at N = 8, 7,500 at N = 10 and 6,500
// at N = 12, with at most 7 % of the launch between them from there to 6,000.
//
// The phases after the row loop deal their tasks over the block's threads in
// order, so that a phase with fewer tasks than threads leaves whole warps idle
// instead of lanes of every warp: the two FP64 sincospi of every region share a
// warp (one such task in every warp took 40 % of the FP64 pipe, 13 % now), the
// moments pair two cells per task, the transforms and the pair sums pair the
// fine and the coarse rule.
template <int N> struct FfShape;
template <> struct FfShape<4> { static constexpr int R = 12, Rn = 6, B = 7; };   // 64 threads
template <> struct FfShape<6> { static constexpr int R = 9, Rn = 3, B = 9; };    // 64
template <> struct FfShape<8> { static constexpr int R = 14, Rn = 6, B = 5; };   // 128
template <> struct FfShape<10> { static constexpr int R = 14, Rn = 5, B = 4; };  // 160
template <> struct FfShape<12> { static constexpr int R = 12, Rn = 4, B = 4; };  // 160
template <int N>
struct FfThreads {
    static constexpr int T = (FfShape<N>::R * (N + 1) + 31) / 32 * 32;
};

// One region's shared memory.  A packed pair of float-float numbers is stored
// as float4 (hi.x, hi.y, lo.x, lo.y).  What both splits keep:
struct FfCommon {
    float4 G[5][5];                  // Fourier moments (fine in lane x, coarse in lane y)
    float2 C[4];                     // sin, cos of the region centre (x, y) times pi
    float2 Q[4];                     // cos qx, sin qx, cos qy, sin qy (flow: of q/2)
    float2 H[2];                     // 1/2T, T (Omega for the flow kinds)
    const int32_t* lm;
    const float4* first;             // table of x1 and exp(-|x1|) at the nodes, or null
    uint32_t pos;
    int L, kind, P;
};
struct FfProducts {
    float4 M[9][9];                  // the product moments M[ac][bd] (fine, coarse)
    float4 T[9][5];                  // G with the x index taken to X_ac
};
template <int N>
struct FfSums {
    float2 Rf[2 * N + 1][5];         // row sums with the row's fine weight
    float2 Rc[N + 1][5];             // coarse (even rows)
};
template <int N>
struct FfColumns {
    float2 Yf[2 * N + 1][5];         // wf_j phi_v(ky_j)
    float2 CY[2 * N + 1][2];         // cos ky, cos ky' (flow kinds: cos(ky -+ qy/2))
    float Yc[N + 1][2][6];           // wc_j phi_v(ky_2j): the five hi words, the lo words
};
template <int N>
struct FfRowsRegion : FfCommon {
    struct Basis { float2 X[2 * N + 1][5]; union { FfColumns<N> col; FfSums<N> sum; }; };
    union {
        Basis a;                     // X = phi_u(kx_i); the column data, then the row sums
        FfProducts b;                // then, from the Fourier moments, the products
    };
    __device__ auto X() { return a.X; }
    __device__ FfColumns<N>& col() { return a.col; }
    __device__ FfSums<N>& sum() { return a.sum; }
};
template <int N>
struct FfNodesRegion : FfCommon {
    float2 x[2 * N + 1][5];
    FfColumns<N> c;
    union {
        float4 AB[N + 1][4];         // A1, B1, A2, B2 of a row pair until F is done
        FfSums<N> s;                 // then the row sums
    };
    union {
        float4 F[N + 1][2 * N + 1];  // the kernel at the nodes of a row pair
        FfProducts b;                // then the products
    };
    __device__ auto X() { return x; }
    __device__ FfColumns<N>& col() { return c; }
    __device__ FfSums<N>& sum() { return s; }
};
template <int N>
struct FfHead {
    float2 tab[64];                  // 2^(j/64)
    float2 wr[2 * N + 1];            // fine weights
    float2 wrc[N + 1];               // coarse weights
    float2 lat[3];                   // -2t, -4t', mu
};
template <int N>
struct FfSmem {
    static constexpr int kHead = (int(sizeof(FfHead<N>)) + 15) / 16 * 16;
    // consecutive regions of the rows split 16 bytes past a multiple of 128
    // apart, so that the regions of one warp read their columns from different banks
    static constexpr int kRow = int(sizeof(FfRowsRegion<N>) + (144 - sizeof(FfRowsRegion<N>) % 128) % 128);
    static constexpr int kNode = int(sizeof(FfNodesRegion<N>));
    static constexpr int kRows = FfShape<N>::R * kRow, kNodes = FfShape<N>::Rn * kNode;
    static constexpr int kBytes = kHead + (kRows > kNodes ? kRows : kNodes);
    static_assert(kRow % 16 == 0 && kNode % 16 == 0, "regions keep 16-byte alignment");
};

__device__ __forceinline__ float4 w_st(w2 a) { return make_float4(a.hi.x, a.hi.y, a.lo.x, a.lo.y); }
__device__ __forceinline__ w2 w_ld(float4 v)
{
    return {make_float2(v.x, v.y), make_float2(v.z, v.w)};
}
// (c, s) rotated by the angle with cosine co and sine so
__device__ __forceinline__ void w_rot(w2 c, w2 s, w2 co, w2 so, w2& c2, w2& s2)
{
    c2 = w_sub(w_mul(c, co), w_mul(s, so));
    s2 = w_add(w_mul(s, co), w_mul(c, so));
}

// Coefficients g_u of a function in the basis phi = (1, c, s, cos 2k, sin 2k)
// (c, s = cos k, sin k) to its products with (1, c, s) x (1, c', s'), index
// 3a + c, where (c', s') is (c, sg s) rotated by the angle with cosine cq and
// sine sq (sg = -1 for pp's k' = q - k).  With c^2 = (1 + cos 2k) / 2,
// s^2 = (1 - cos 2k) / 2 and s c = sin 2k / 2:
//   c'   = cq c - sg sq s           s'   = sq c + sg cq s
//   c c' = cq (1 + cos 2k)/2 - sg sq sin 2k/2
//   c s' = sq (1 + cos 2k)/2 + sg cq sin 2k/2
//   s c' = cq sin 2k/2 - sg sq (1 - cos 2k)/2
//   s s' = sq sin 2k/2 + sg cq (1 - cos 2k)/2
// Product k goes to o[k * stride] as it is formed.
__device__ __forceinline__ void w_fourier_to_products(const w2 g[5], float2 cq1, float2 sq1,
                                                      bool flip, float4* o, int stride)
{
    const w2 cq = w_dup(cq1), sq = w_dup(sq1);
    const w2 cs = flip ? w_neg(cq) : cq, ss = flip ? w_neg(sq) : sq;   // sg cq, sg sq
    const w2 hc = w_scale(0.5f, cq), hs = w_scale(0.5f, sq);
    const w2 hcs = w_scale(0.5f, cs), hss = w_scale(0.5f, ss);
    const w2 pl = w_add(g[0], g[3]), mi = w_sub(g[0], g[3]);
    o[0 * stride] = w_st(g[0]);
    o[1 * stride] = w_st(w_sub(w_mul(cq, g[1]), w_mul(ss, g[2])));
    o[2 * stride] = w_st(w_add(w_mul(sq, g[1]), w_mul(cs, g[2])));
    o[3 * stride] = w_st(g[1]);
    o[4 * stride] = w_st(w_sub(w_mul(hc, pl), w_mul(hss, g[4])));
    o[5 * stride] = w_st(w_add(w_mul(hs, pl), w_mul(hcs, g[4])));
    o[6 * stride] = w_st(g[2]);
    o[7 * stride] = w_st(w_sub(w_mul(hc, g[4]), w_mul(hss, mi)));
    o[8 * stride] = w_st(w_add(w_mul(hs, g[4]), w_mul(hcs, mi)));
}

// The phases of a block on `live` regions (entries t0 ... of the eval list),
// region r at reg(r).  KF: the kinds the launch may meet -- 0 any, 1 no flow
// kind, 2 flow kinds only -- so that a launch carries only the kernel F it needs
// (the row loop's code stays within the instruction cache).
template <int KF>
__device__ __forceinline__ bool ff_flow(int kind) { return KF == 2 || (KF == 0 && is_flow(kind)); }

// the per-region inputs: the exact dyadic centre / pi = -1 + (2 ix + 1) 2^-L (x,
// then y) by the first threads, the transfer momentum and the temperature by
// those from kIn on
template <int kIn, class Reg, class Entry>
__device__ __forceinline__ void ff_inputs(const Work& w, int cur, int live, Reg reg, Entry entry)
{
    const int tid = threadIdx.x;
    if (tid < 2 * live) {
        FfCommon& E = reg(tid >> 1);
        const uint64_t key = w.key[cur][w.evl[entry(tid >> 1)].x];
        const int i = tid & 1;
        const uint32_t ic = i == 0 ? key_ix(key) : key_iy(key);
        double sn, cs;
        sincospi(fma(double(2 * ic + 1), ldexp(1.0, -int(key_level(key))), -1.0), &sn, &cs);
        E.C[2 * i] = ff_st(ff_from(sn));
        E.C[2 * i + 1] = ff_st(ff_from(cs));
    } else if (tid >= kIn && tid - kIn < live) {
        FfCommon& E = reg(tid - kIn);
        const uint2 e = w.evl[entry(tid - kIn)];
        const uint32_t mt = w.meta[e.y];
        const QTrig tq = w.trig[e.y];     // flow kinds: rotation by q/2
        const DevBatch& B = w.batches[meta_batch(mt)];
        E.Q[0] = ff_st(ff_from(tq.cqx));
        E.Q[1] = ff_st(ff_from(tq.sqx));
        E.Q[2] = ff_st(ff_from(tq.cqy));
        E.Q[3] = ff_st(ff_from(tq.sqy));
        E.H[0] = ff_st(ff_from(B.inv2T));
        E.H[1] = ff_st(ff_from(B.T));
        E.lm = B.lm;
        E.pos = e.x;
        E.L = int(key_level(w.key[cur][e.x]));
        E.kind = meta_kind(mt);
        E.P = B.npairs;
    }
}

// Rows and columns ra = 2 ei, rb = ra + 1 of the fine grid (the last pair
// carries its one row in both lanes): the basis at both into D, and the rows'
// energies e = A + B cos ky along the row for k and for k', in units of 2T
template <int N, int KF, class Region>
__device__ __forceinline__ void ff_basis(Region& D, const FfHead<N>& S, int ei, w2& A1, w2& B1,
                                         w2& A2, w2& B2)
{
    const int v = rule_variant(N);
    const int ra = 2 * ei, rb = ei < N ? 2 * ei + 1 : 2 * N;
    const int kind = D.kind;
    const bool pp = kind == PP, flow = ff_flow<KF>(kind);
    const float4 ta = g_cosine[v][D.L][ra <= N ? ra : 2 * N - ra];
    const float4 tb = g_cosine[v][D.L][rb <= N ? rb : 2 * N - rb];
    const float2 sgn = make_float2(ra <= N ? 1.0f : -1.0f, rb <= N ? 1.0f : -1.0f);
    const w2 co = w_pair(make_float2(ta.x, ta.y), make_float2(tb.x, tb.y));
    const w2 so = w_flip(w_pair(make_float2(ta.z, ta.w), make_float2(tb.z, tb.w)), sgn);
    const w2 cqx = w_dup(D.Q[0]), sqx = w_dup(D.Q[1]);
    const w2 cqy = w_dup(D.Q[2]), sqy = w_dup(D.Q[3]);
    w2 cx, sx, cy, sy;
    w_rot(w_dup(D.C[1]), w_dup(D.C[0]), co, so, cx, sx);
    w_rot(w_dup(D.C[3]), w_dup(D.C[2]), co, so, cy, sy);
    // the Fourier basis there
    auto X = D.X();
    FfColumns<N>& Y = D.col();
    const w2 wf = w_pair(S.wr[ra], S.wr[rb]), wc = w_dup(S.wrc[ei]);
    auto put_x = [&](int u, w2 p) {
        X[ra][u] = w_x(p);
        X[rb][u] = w_y(p);
    };
    auto put_y = [&](int u, w2 p) {
        const w2 f = w_mul(wf, p);
        Y.Yf[ra][u] = w_x(f);
        Y.Yf[rb][u] = w_y(f);
        const w2 c = w_mul(wc, {dup(p.hi.x), dup(p.lo.x)});   // the even column, in both lanes
        Y.Yc[ei][0][u] = c.hi.x;
        Y.Yc[ei][1][u] = c.lo.x;
    };
    put_x(0, w_dup(1.0f, 0.0f));
    put_x(1, cx);
    put_x(2, sx);
    put_x(3, w_mul(w_sub(cx, sx), w_add(cx, sx)));
    put_x(4, w_mul(w_scale(2.0f, sx), cx));
    put_y(0, w_dup(1.0f, 0.0f));
    put_y(1, cy);
    put_y(2, sy);
    put_y(3, w_mul(w_sub(cy, sy), w_add(cy, sy)));
    put_y(4, w_mul(w_scale(2.0f, sy), cy));
    Y.Yc[ei][0][5] = 0.0f;
    Y.Yc[ei][1][5] = 0.0f;
    const w2 tA = w_dup(S.lat[0]), tB = w_dup(S.lat[1]), nmu = w_neg(w_dup(S.lat[2]));
    // the shifted k' (q + k: rotate by q; q - k: rotate -k by q); flow kinds:
    // e(k + q/2) and e(k - q/2), Q the rotation by q/2
    w2 cx1 = cx, cx2, cy1 = cy, cy2, sn;
    if (flow) {
        w_rot(cx, sx, cqx, sqx, cx1, sn);
        w_rot(cx, sx, cqx, w_neg(sqx), cx2, sn);
        w_rot(cy, sy, cqy, sqy, cy1, sn);
        w_rot(cy, sy, cqy, w_neg(sqy), cy2, sn);
    } else {
        w_rot(cx, pp ? w_neg(sx) : sx, cqx, sqx, cx2, sn);
        w_rot(cy, pp ? w_neg(sy) : sy, cqy, sqy, cy2, sn);
    }
    Y.CY[ra][0] = w_x(cy1);
    Y.CY[rb][0] = w_y(cy1);
    Y.CY[ra][1] = w_x(cy2);
    Y.CY[rb][1] = w_y(cy2);
    A1 = w_fma(tA, cx1, nmu);
    B1 = w_fma(tB, cx1, tA);
    A2 = w_fma(tA, cx2, nmu);
    B2 = w_fma(tB, cx2, tA);
    if (flow) {
        // pp: minus the divided difference at (e1, -e2); the leading sign goes
        // into the row weights
        if (kind == FLOW_PP) { A2 = w_neg(A2); B2 = w_neg(B2); }
    } else {
        // x = e / 2T (for pp the second energy enters with its sign flipped)
        const w2 h1 = w_dup(D.H[0]), h2 = pp ? w_neg(h1) : h1;
        A1 = w_mul(A1, h1);
        B1 = w_mul(B1, h1);
        A2 = w_mul(A2, h2);
        B2 = w_mul(B2, h2);
    }
}

// the kernel F at column j of a row pair
template <int KF, class Region>
__device__ __forceinline__ w2 ff_node(const Region& D, const float2 cy[2], w2 A1, w2 B1, w2 A2,
                                      w2 B2, const float2* tab)
{
    const w2 x1 = w_fma(B1, w_dup(cy[0]), A1);
    const w2 x2 = w_fma(B2, w_dup(cy[1]), A2);
    if (KF != 1 && is_flow(D.kind)) return w_flow_Fdot(x1, x2, w_dup(D.H[1]));
    if (KF != 2 && D.kind != OVERLAP)
        return w_bubble_F2T(x1, w_exp_neg(w_abs(x1), tab), x2, tab);
    return w_dup(1.0f, 0.0f);
}

// a row pair's weight (flow pp: with the kind's leading sign) on its normalised sum
template <int KF>
__device__ __forceinline__ w2 ff_weigh(int kind, w2 wr, w2 sum)
{
    if (KF != 1 && kind == FLOW_PP) wr = w_neg(wr);
    return w_mul(wr, w_fast(sum.hi, sum.lo));
}

// From the row sums: Fourier moments, product moments, every pair's values
template <int N, int KF, class Reg>
__device__ __forceinline__ void ff_finish(const Work& w, int cur, int64_t t0, int live, Reg reg,
                                          double* rule_q2, double* rule_d)
{
    constexpr int NF = 2 * N + 1, kThreads = FfThreads<N>::T;
    const int tid = threadIdx.x;
    // Fourier moments G[u][v], float-float dot products over the rows: cells c
    // and c + 13 of the 25 in the two lanes
    for (int k = tid; k < 13 * live; k += kThreads) {
        auto& E = reg(k / 13);
        auto X = E.X();
        const FfSums<N>& R = E.sum();
        const int ca = k % 13, cb = ca + 13 < 25 ? ca + 13 : ca;
        const int ua = ca / 5, va = ca - 5 * ua, ub = cb / 5, vb = cb - 5 * ub;
        w2 gf = w_zero(), gc = w_zero();
#pragma unroll 5
        for (int r = 0; r < NF; ++r)
            w_acc(w_pair(X[r][ua], X[r][ub]), w_pair(R.Rf[r][va], R.Rf[r][vb]), gf);
#pragma unroll 4
        for (int r = 0; r <= N; ++r)
            w_acc(w_pair(X[2 * r][ua], X[2 * r][ub]), w_pair(R.Rc[r][va], R.Rc[r][vb]), gc);
        gf = w_fast(gf.hi, gf.lo);
        gc = w_fast(gc.hi, gc.lo);
        E.G[ua][va] = make_float4(gf.hi.x, gc.hi.x, gf.lo.x, gc.lo.x);
        E.G[ub][vb] = make_float4(gf.hi.y, gc.hi.y, gf.lo.y, gc.lo.y);
    }
    __syncthreads();
    // the rotation of k' and its orientation: (cos q, sin q) per direction for
    // ph / pp (pp: k' = q - k), none for the flow kinds (both form factors at k)
    const float2 one = make_float2(1.0f, 0.0f), zero = make_float2(0.0f, 0.0f);
    // x: each column v of G to the nine X_ac
    for (int k = tid; k < 5 * live; k += kThreads) {
        auto& E = reg(k / 5);
        const int vc = k % 5;
        const bool fl = ff_flow<KF>(E.kind);
        w2 g[5];
#pragma unroll
        for (int u = 0; u < 5; ++u) g[u] = w_ld(E.G[u][vc]);
        w_fourier_to_products(g, fl ? one : E.Q[0], fl ? zero : E.Q[1], !fl && E.kind == PP,
                              &E.b.T[0][vc], 5);
    }
    __syncthreads();
    // y: each row ac to the nine Y_bd
    for (int k = tid; k < 9 * live; k += kThreads) {
        auto& E = reg(k / 9);
        const int ac = k % 9;
        const bool fl = ff_flow<KF>(E.kind);
        w2 g[5];
#pragma unroll
        for (int u = 0; u < 5; ++u) g[u] = w_ld(E.b.T[ac][u]);
        w_fourier_to_products(g, fl ? one : E.Q[2], fl ? zero : E.Q[3], !fl && E.kind == PP,
                              &E.b.M[ac][0], 1);
    }
    __syncthreads();
    for (int k = tid; k < kGroupPairs * live; k += kThreads) {
        auto& E = reg(k / kGroupPairs);
        const int p = k % kGroupPairs, P = E.P, kind = E.kind;
        if (p >= P) continue;
        // the Jacobian: 1/2T (ph, pp) in float-float times 4^-L / 4, an exact
        // power of two applied to both words
        const w2 jac = kind == PH || kind == PP ? w_dup(E.H[0]) : w_dup(one);
        const float p2 = __int_as_float((125 - 2 * E.L) << 23);
        const int l = E.lm[2 * p], m = E.lm[2 * p + 1];
        w2 q = w_zero();               // Q_2N, Q_N
        if (l >= 0 && m >= 0 && l < w.nff && m < w.nff) {
            const float4* term = g_terms[l][m];
            for (int t = 0; t < 4; ++t) {
                const float4 c = term[t];
                if (__float_as_int(c.z) < 0) break;
                w_acc(w_dup(c.x, c.y), w_ld((&E.b.M[0][0])[__float_as_int(c.z)]), q);
            }
        }
        q = w_fast(q.hi, q.lo);
        // Q_2N and the embedded-rule difference Q_N - Q_2N; only the value's
        // conversion to FP64 leaves the FP32 pipe
        const w2 base = {make_float2(0.0f, q.hi.x), make_float2(0.0f, q.lo.x)};
        const w2 r = w_mul(w_sub(q, base), jac);
        const float2 hi = mul2(r.hi, dup(p2)), lo = mul2(r.lo, dup(p2));
        const double v2 = double(hi.x) + double(lo.x);
        if (rule_q2) {
            const int64_t o = (t0 + k / kGroupPairs) * P + p;
            rule_q2[o] = v2;
            rule_d[o] = double(hi.y) + double(lo.y);
        } else {
            const size_t o = size_t(E.pos) * size_t(w.vstride) + size_t(p);
            w.vval[cur][o] = v2;
            w.verr[cur][o] = fabsf(hi.y);
        }
    }
}

// the table blocks: a task per row pair for the basis, then one per column of it (as
// the nodes split, so that few regions spread over the device)
template <int N>
__global__ void __launch_bounds__(FfThreads<N>::T, FfShape<N>::B) k_first_eval(Work w, Lattice lat)
{
    constexpr int NF = 2 * N + 1, RP = N + 1, kThreads = FfThreads<N>::T;
    constexpr int kIn = (2 * FfShape<N>::Rn + 31) / 32 * 32;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    const RoundCounts rc = round_counts(w);
    if (!first_sharing(w, rc.n)) return;
    FfHead<N>& S = *reinterpret_cast<FfHead<N>*>(smem_raw);
    FfNodesRegion<N>* const regions =
        reinterpret_cast<FfNodesRegion<N>*>(smem_raw + FfSmem<N>::kHead);
    auto reg = [&](int r) -> FfNodesRegion<N>& { return regions[r]; };
    const First f = first_view<N>(w);
    const bool used = first_used<N, true>(rc, f);
    note_sharing(w, rc, used, f.room);
    if (!used) return;
    const int cur = w.ls->cur, tid = threadIdx.x, v = rule_variant(N);
    const uint32_t count = uint32_t(rc.distinct);
    const uint32_t share = (count + gridDim.x - 1) / gridDim.x;
    const uint32_t R = min(share, uint32_t(FfShape<N>::Rn));
    if (blockIdx.x * R >= count) return;
    for (int k = tid; k < 64; k += kThreads) S.tab[k] = ff_st(ff_from(c_exp2d[k]));
    if (tid < NF) S.wr[tid] = ff_st(ff_from(c_wf[v][tid]));
    if (tid <= N) S.wrc[tid] = ff_st(ff_from(c_wc[v][tid]));
    if (tid < 3)
        S.lat[tid] = ff_st(ff_from(tid == 0 ? -2.0 * lat.t : tid == 1 ? -4.0 * lat.tp : lat.mu));
    for (uint32_t u0 = blockIdx.x * R; u0 < count; u0 += gridDim.x * R) {
        const int live = int(min(R, count - u0));
        ff_inputs<kIn>(w, cur, live, reg, [&](int r) { return f.rep[u0 + r]; });
        __syncthreads();
        for (int k = tid; k < RP * live; k += kThreads) {
            FfNodesRegion<N>& D = reg(k / RP);
            w2 A1, B1, A2, B2;
            ff_basis<N, 1>(D, S, k % RP, A1, B1, A2, B2);
            D.AB[k % RP][0] = w_st(A1);
            D.AB[k % RP][1] = w_st(B1);
        }
        __syncthreads();
#pragma unroll 1
        for (int k = tid; k < RP * NF * live; k += kThreads) {
            const int r = k / (RP * NF), node = k % (RP * NF), j = node / RP, ei = node - RP * j;
            FfNodesRegion<N>& D = reg(r);
            const w2 x1 = w_fma(w_ld(D.AB[ei][1]), w_dup(D.c.CY[j][0]), w_ld(D.AB[ei][0]));
            float4* out = first_block(f, u0 + r) + node;
            out[0] = w_st(x1);
            out[RP * NF] = w_st(w_exp_neg(w_abs(x1), S.tab));
        }
        __syncthreads();
    }
}

template <int N, int KF>
__global__ void __launch_bounds__(FfThreads<N>::T, FfShape<N>::B)
k_eval_group_ff(Work w, Lattice lat, double* rule_q2, double* rule_d)
{
    constexpr int NF = 2 * N + 1, RP = N + 1, kThreads = FfThreads<N>::T;
    constexpr int kIn = (2 * FfShape<N>::R + 31) / 32 * 32;
    static_assert(FfShape<N>::Rn <= FfShape<N>::R && kIn + FfShape<N>::R <= kThreads,
                  "region inputs: one thread each");
    extern __shared__ __align__(16) unsigned char smem_raw[];
    FfHead<N>& S = *reinterpret_cast<FfHead<N>*>(smem_raw);
    unsigned char* const smem = smem_raw + FfSmem<N>::kHead;
    const int cur = w.ls->cur, tid = threadIdx.x;
    const int64_t n_eval = w.ls->n_eval;
    const bool nodes = n_eval <= kNodesMax;
    const int64_t share = (n_eval + gridDim.x - 1) / gridDim.x;
    const int R = !nodes ? FfShape<N>::R : int(share < FfShape<N>::Rn ? share : FfShape<N>::Rn);
    if (int64_t(blockIdx.x) * R >= n_eval) return;
    const int v = rule_variant(N);
    for (int k = tid; k < 64; k += kThreads) S.tab[k] = ff_st(ff_from(c_exp2d[k]));
    if (tid < NF) S.wr[tid] = ff_st(ff_from(c_wf[v][tid]));
    if (tid <= N) S.wrc[tid] = ff_st(ff_from(c_wc[v][tid]));
    if (tid < 3)
        S.lat[tid] = ff_st(ff_from(tid == 0 ? -2.0 * lat.t : tid == 1 ? -4.0 * lat.tp : lat.mu));

    if (nodes) {
        auto reg = [&](int r) -> FfNodesRegion<N>& {
            return reinterpret_cast<FfNodesRegion<N>*>(smem)[r];
        };
        for (int64_t t0 = int64_t(blockIdx.x) * R; t0 < n_eval; t0 += int64_t(gridDim.x) * R) {
            const int live = int(n_eval - t0 < R ? n_eval - t0 : R);
            ff_inputs<kIn>(w, cur, live, reg, [&](int r) { return t0 + r; });
            __syncthreads();
            for (int k = tid; k < RP * live; k += kThreads) {
                FfNodesRegion<N>& D = reg(k / RP);
                w2 A1, B1, A2, B2;
                ff_basis<N, KF>(D, S, k % RP, A1, B1, A2, B2);
                float4* ab = D.AB[k % RP];
                ab[0] = w_st(A1);
                ab[1] = w_st(B1);
                ab[2] = w_st(A2);
                ab[3] = w_st(B2);
            }
            __syncthreads();
#pragma unroll 1
            for (int k = tid; k < RP * NF * live; k += kThreads) {
                FfNodesRegion<N>& D = reg(k / (RP * NF));
                const int node = k % (RP * NF), ei = node / NF, j = node - NF * ei;
                const float4* ab = D.AB[ei];
                D.F[ei][j] = w_st(ff_node<KF>(D, D.c.CY[j], w_ld(ab[0]), w_ld(ab[1]), w_ld(ab[2]),
                                              w_ld(ab[3]), S.tab));
            }
            __syncthreads();
            // row sums in column order: fine sums of two rows (one per lane), then
            // coarse sums of an even row, two of the five in a pair
            for (int k = tid; k < 8 * RP * live; k += kThreads) {
                if (k < 5 * RP * live) {
                    FfNodesRegion<N>& D = reg(k / (5 * RP));
                    const int t = k % (5 * RP), ei = t / 5, u = t - 5 * ei;
                    const int ra = 2 * ei, rb = ei < N ? 2 * ei + 1 : 2 * N;
                    w2 rf = w_zero();
#pragma unroll 5
                    for (int j = 0; j < NF; ++j) w_acc(w_ld(D.F[ei][j]), w_dup(D.c.Yf[j][u]), rf);
                    const w2 f = ff_weigh<KF>(D.kind, w_pair(S.wr[ra], S.wr[rb]), rf);
                    D.s.Rf[ra][u] = w_x(f);
                    D.s.Rf[rb][u] = w_y(f);
                } else {
                    const int kc = k - 5 * RP * live;
                    FfNodesRegion<N>& D = reg(kc / (3 * RP));
                    const int t = kc % (3 * RP), ei = t / 3, u = t - 3 * ei;
                    w2 rc = w_zero();
#pragma unroll 4
                    for (int j = 0; j <= N; ++j) {
                        const float4 F = D.F[ei][2 * j];
                        w_acc(w_dup(F.x, F.z),
                              {*reinterpret_cast<const float2*>(&D.c.Yc[j][0][2 * u]),
                               *reinterpret_cast<const float2*>(&D.c.Yc[j][1][2 * u])}, rc);
                    }
                    const w2 c = ff_weigh<KF>(D.kind, w_dup(S.wrc[ei]), rc);
                    D.s.Rc[ei][2 * u] = w_x(c);
                    if (u < 2) D.s.Rc[ei][2 * u + 1] = w_y(c);
                }
            }
            __syncthreads();
            ff_finish<N, KF>(w, cur, t0, live, reg, rule_q2, rule_d);
            __syncthreads();
        }
        return;
    }

    auto reg = [&](int r) -> FfRowsRegion<N>& {
        return *reinterpret_cast<FfRowsRegion<N>*>(smem + r * FfSmem<N>::kRow);
    };
    const RoundCounts rc = round_counts(w);
    const First fs = KF != 2 && first_sharing(w, rc.n) ? first_view<N>(w) : First{};
    const bool first = KF != 2 && first_sharing(w, rc.n) && first_used<N, true>(rc, fs);
    // this thread's region and rows (threads past the last row pair have none)
    const int rho = tid / RP, ei = tid % RP;
    const int ra = 2 * ei, rb = ei < N ? 2 * ei + 1 : 2 * N;
    for (int64_t t0 = int64_t(blockIdx.x) * R; t0 < n_eval; t0 += int64_t(gridDim.x) * R) {
        const int live = int(n_eval - t0 < R ? n_eval - t0 : R);
        ff_inputs<kIn>(w, cur, live, reg, [&](int r) { return t0 + r; });
        if (KF != 2 && first && tid >= kIn && tid - kIn < live)
            reg(tid - kIn).first = first_find(fs, t0 + tid - kIn);
        __syncthreads();
        FfRowsRegion<N>& D = reg(rho < live ? rho : 0);
        w2 A1, B1, A2, B2;
        if (rho < live) ff_basis<N, KF>(D, S, ei, A1, B1, A2, B2);
        // with every region's first energy known, a loop without it
        const bool known = __syncthreads_and(KF != 2 && first && (rho >= live || D.first));
        // fine sums of both rows (one per lane); coarse sums of the even row, two
        // of the five in a pair
        w2 rf[5], rc[3];
#pragma unroll
        for (int k = 0; k < 5; ++k) rf[k] = w_zero();
#pragma unroll
        for (int k = 0; k < 3; ++k) rc[k] = w_zero();
        if (rho < live) {
            const FfColumns<N>& Y = D.a.col;
            auto sums = [&](int j, w2 F) {
#pragma unroll
                for (int k = 0; k < 5; ++k) w_acc(F, w_dup(Y.Yf[j][k]), rf[k]);
                if ((j & 1) == 0) {
                    const w2 Fe = {dup(F.hi.x), dup(F.lo.x)};
#pragma unroll
                    for (int k = 0; k < 3; ++k)
                        w_acc(Fe, {*reinterpret_cast<const float2*>(&Y.Yc[j >> 1][0][2 * k]),
                                   *reinterpret_cast<const float2*>(&Y.Yc[j >> 1][1][2 * k])}, rc[k]);
                }
            };
            // not unrolled: a node is some 500 instructions, and an unrolled row
            // overflows the instruction cache
            if (KF != 2 && known) {
                const float4* at = D.first + ei;
                float4 nx = __ldg(at), nv = __ldg(at + RP * NF);   // one column ahead
#pragma unroll 1
                for (int j = 0; j < NF; ++j) {
                    const w2 x1 = w_ld(nx), v1 = w_ld(nv);
                    at += j + 1 < NF ? RP : 0;
                    nx = __ldg(at);
                    nv = __ldg(at + RP * NF);
                    sums(j, w_bubble_F2T(x1, v1, w_fma(B2, w_dup(Y.CY[j][1]), A2), S.tab));
                }
            } else {
#pragma unroll 1
                for (int j = 0; j < NF; ++j)
                    sums(j, ff_node<KF>(D, Y.CY[j], A1, B1, A2, B2, S.tab));
            }
        }
        // the row sums take the column data's memory: every row is done first
        __syncthreads();
        if (rho < live) {
#pragma unroll
            for (int k = 0; k < 5; ++k) {
                const w2 f = ff_weigh<KF>(D.kind, w_pair(S.wr[ra], S.wr[rb]), rf[k]);
                D.a.sum.Rf[ra][k] = w_x(f);
                D.a.sum.Rf[rb][k] = w_y(f);
            }
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const w2 c = ff_weigh<KF>(D.kind, w_dup(S.wrc[ei]), rc[k]);
                D.a.sum.Rc[ei][2 * k] = w_x(c);
                if (k < 2) D.a.sum.Rc[ei][2 * k + 1] = w_y(c);
            }
        }
        __syncthreads();
        ff_finish<N, KF>(w, cur, t0, live, reg, rule_q2, rule_d);
        __syncthreads();
    }
}

template <int N>
static cudaError_t group_attr()
{
    cudaError_t e = cudaFuncSetAttribute(k_eval_group<N>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         int(sizeof(GroupSmem<N>)));
    for (int kf = 0; kf < 3 && e == cudaSuccess; ++kf)
        e = cudaFuncSetAttribute(kf == 0 ? k_eval_group_ff<N, 0>
                                 : kf == 1 ? k_eval_group_ff<N, 1> : k_eval_group_ff<N, 2>,
                                 cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 FfSmem<N>::kBytes);
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_first_eval<N>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 FfSmem<N>::kBytes);
    return e;
}

static cudaError_t group_kernel_attributes()
{
    cudaError_t e = group_attr<4>();
    if (e == cudaSuccess) e = group_attr<6>();
    if (e == cudaSuccess) e = group_attr<8>();
    if (e == cudaSuccess) e = group_attr<10>();
    if (e == cudaSuccess) e = group_attr<12>();
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_eval_df<6, true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 DfColumns<6, true>::kBytes);
    return e;
}

int share_kernels(const Work& w, int64_t hint_eval, int fp32)
{
    if (!w.share || hint_eval <= 0) return 0;
    if (w.vstride > 0) return hint_eval > kNodesMax ? 3 : 0;
    return fp32 ? 4 : 3;   // float-float: with and without the tables
}

template <int N>
static void group_launch(const Work& w, int64_t hint_eval, int64_t cap, int fp32, Lattice lat,
                         cudaStream_t s, double* rule_q2, double* rule_d)
{
    constexpr int R = GroupShape<N>::R;
    const int64_t blocks = std::min<int64_t>((hint_eval + R - 1) / R, cap);
    // a block per R regions; when those are few, up to a resident grid's blocks
    // (152 SMs x B) with fewer regions each (the nodes split)
    const int64_t resident = 152 * FfShape<N>::B;
    const int64_t ff = std::max((hint_eval + FfShape<N>::R - 1) / FfShape<N>::R,
                                std::min(hint_eval, resident));
    const dim3 grid(static_cast<unsigned>(std::min(ff, cap))), block(FfThreads<N>::T);
    const size_t sm = FfSmem<N>::kBytes;
    if (share_kernels(w, hint_eval, fp32)) {
        const int few = int(std::min<int64_t>((hint_eval + 255) / 256, 152 * kInsertBlocks));
        k_first_clear<N><<<few, 256, 0, s>>>(w);
        k_first_insert<N><<<few, 256, 0, s>>>(w);
        if (fp32) k_first_eval<N><<<unsigned(resident), block, sm, s>>>(w, lat);
        else      k_first_eval_fp64<N><<<152 * 8, R * (2 * N + 1), 0, s>>>(w, lat);
    }
    if (fp32 && w.kinds == 1)
        k_eval_group_ff<N, 1><<<grid, block, sm, s>>>(w, lat, rule_q2, rule_d);
    else if (fp32 && w.kinds == 2)
        k_eval_group_ff<N, 2><<<grid, block, sm, s>>>(w, lat, rule_q2, rule_d);
    else if (fp32)
        k_eval_group_ff<N, 0><<<grid, block, sm, s>>>(w, lat, rule_q2, rule_d);
    else
        k_eval_group<N><<<int(blocks), R * (2 * N + 1), sizeof(GroupSmem<N>), s>>>(
            w, lat, rule_q2, rule_d);
}

cudaError_t launch_eval_group(const Work& w, int64_t hint_eval, int rule_n, int fp32, Lattice lat,
                              cudaStream_t s, double* rule_q2, double* rule_d, int max_blocks)
{
    if (hint_eval <= 0) return cudaSuccess;
    const int64_t cap = max_blocks > 0 ? max_blocks : 152 * 32;
    switch (rule_n) {
    case 4: group_launch<4>(w, hint_eval, cap, fp32, lat, s, rule_q2, rule_d); break;
    case 6: group_launch<6>(w, hint_eval, cap, fp32, lat, s, rule_q2, rule_d); break;
    case 8: group_launch<8>(w, hint_eval, cap, fp32, lat, s, rule_q2, rule_d); break;
    case 10: group_launch<10>(w, hint_eval, cap, fp32, lat, s, rule_q2, rule_d); break;
    default: group_launch<12>(w, hint_eval, cap, fp32, lat, s, rule_q2, rule_d); break;
    }
    return cudaGetLastError();
}

cudaError_t launch_eval(const Work& w, int64_t hint_eval, int rule_n, int fp32, Lattice lat,
                        cudaStream_t s, cudaEvent_t mid)
{
    if (hint_eval <= 0) return cudaSuccess;
    const int threads = 128;
    int64_t blocks = (hint_eval + threads - 1) / threads;
    if (blocks > 152 * 64) blocks = 152 * 64;
    if (w.share) {
        if (rule_n == 4) fp32 ? share_launch<4, true>(w, hint_eval, lat, s)
                              : share_launch<4, false>(w, hint_eval, lat, s);
        else             fp32 ? share_launch<6, true>(w, hint_eval, lat, s)
                              : share_launch<6, false>(w, hint_eval, lat, s);
    }
    if (fp32) {
        if (rule_n == 4) k_eval_fp32<4><<<int(blocks), threads, 0, s>>>(w, lat);
        else             k_eval_fp32<6><<<int(blocks), threads, 0, s>>>(w, lat);
        if (mid) {
            const cudaError_t e = cudaEventRecord(mid, s);
            if (e != cudaSuccess) return e;
        }
        if (w.share) rule_n == 4 ? df_launch<4, true>(w, hint_eval, lat, s)
                                 : df_launch<6, true>(w, hint_eval, lat, s);
        rule_n == 4 ? df_launch<4, false>(w, hint_eval, lat, s)
                    : df_launch<6, false>(w, hint_eval, lat, s);
    } else {
        if (rule_n == 4) k_eval_fp64<4><<<int(blocks), threads, 0, s>>>(w, lat);
        else             k_eval_fp64<6><<<int(blocks), threads, 0, s>>>(w, lat);
    }
    return cudaGetLastError();
}

}  // namespace paid
