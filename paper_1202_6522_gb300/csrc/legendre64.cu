// legendre64.cu -- the FP64 Legendre stage on the CUDA cores, scalar and vector.
//
// The sums and the mirror folding are those of legendre.cu; this file holds
// what FP64 asks for on this GPU.  Its FP64 pipe takes one warp instruction
// every ~19 cycles per SM (every ~64 per SM quarter), some seventy times fewer
// than FP32, so a kernel's time is its count of FP64 instructions, provided
// every SM quarter has a warp with work.
//
// * Recurrence in two instructions instead of three.  Within a segment of
//   kSeedSeg degrees P_n^m = s_n Q_n with s_n = prod a_j over the segment's
//   degrees up to n, and Q_n = x Q_{n-1} + beta_n Q_{n-2}, beta_n = b_n / (a_n a_{n-1})
//   = -((n-1)^2 - m^2) / (4 (n-1)^2 - 1) (Sec. 3.2 divided by s_n; beta = b_n / a_n
//   at the segment's first degree, whose two predecessors are the stored state).
//   s_n goes into the spectral value once per degree and field, not per
//   latitude.  A power of two per segment, taken into the stored state, centres
//   the range of s on 1 (2^-70 .. 2^70 at order 2047).
// * Vector transforms are scalar ones.  With eps_n = sqrt((n^2 - m^2) / (4 n^2 - 1)),
//   sin(theta) dP_n/dtheta = n eps_{n+1} P_{n+1} - (n + 1) eps_n P_{n-1}, so
//     sin V_theta = sum_k U_k P_k,  U_k = (k-1) eps_k S_{k-1} - (k+2) eps_{k+1} S_{k+1} - i m T_k,
//     sin V_phi   = sum_k W_k P_k,  W_k = (k-1) eps_k T_{k-1} - (k+2) eps_{k+1} T_{k+1} + i m S_k
//   for k = m .. lmax + 1: per field two complex sums per degree and pair
//   instead of four, and no derivative to generate.  The differences multiply
//   by n whatever is not smooth in n in the errors of P, near the poles above
//   all, so here the recurrence is Sec. 3.2's own, the one whose states are
//   stored (the Q_n agree with them to rounding only and would jump at every
//   segment: errors 1.1 times as large, geometric mean over N = 33 .. 124, up
//   to 5 times; with Sec. 3.2's the errors are those of the form with
//   derivatives).  The analysis is the transpose: A_k, B_k = sum P_k fold(V_theta), fold(V_phi), then
//     S_n = n eps_{n+1} A_{n+1} - (n+1) eps_n A_{n-1} - i m B_n,
//     T_n = n eps_{n+1} B_{n+1} - (n+1) eps_n B_{n-1} + i m A_n.
#include <cuda_runtime.h>

#include "sht_internal.h"

namespace sht {
namespace {

constexpr unsigned kFull = 0xffffffffu;
constexpr double kDown = 0x1p-240;   // 2^-Scale<double>::S
constexpr int kHiOne = 0x3ff00000;   // high word of 1.0
constexpr int kMaxDeg = kSeedSeg + 2;   // degrees of a segment: kSeedSeg, one more at lmax + 1, padded to even

// Orders' first index in a table or spectrum that runs to degree lmax + ext.
__device__ __forceinline__ long col_ext(const PlanView<double> &pv, int m, int ext)
{
    return col_of_mres(pv.lmax + ext, m, pv.mres);
}

// CTAs that are all resident at once go to the SMs round robin; every second
// round of `nsm` runs backwards, so that an SM with a heavy item of one round
// takes a light one of the next (the items come heaviest first).
__device__ __forceinline__ int snake(int i, int total, int nsm)
{
    const int r = i / nsm, first = r * nsm;
    if (!(r & 1)) return i;
    const int len = min(nsm, total - first);
    return first + len - 1 - (i - first);
}

// Spectra of a vector transform's scalar form: the degrees m .. lmax of U (or A) and
// of W (B) as [nb][nlm] each, and the degree lmax + 1 of both as [2 nb][mmax + 1], for
// a group of nb <= kVec64Group fields.  Field f of the scalar form is U of field f,
// then W of field f - nb; its E/O or folds are field f + lo, or f + hi, of the call's.
struct VecSpec {
    double2 *u, *w, *top;
    int nb, lo, hi;
    __device__ __forceinline__ int inter(int f) const { return f + (f < nb ? lo : hi); }
    __device__ __forceinline__ double2 *field(int f, int nlm) const
    {
        return f < nb ? u + (size_t)f * nlm : w + (size_t)(f - nb) * nlm;
    }
};

// (a_n, b_n) of Sec. 3.2 at degree m mres + i, i = 0 .. L (degree lmax + 1), and eps_n.
__device__ double2 plain_ab(const PlanView<double> &pv, int m, int i)
{
    const double dm = m * pv.mres, n = dm + i, n1 = n - 1.0;
    if (i == 0) return make_double2(0.0, 1.0);   // the start value P_m^m, handed over as P_{m-2}
    if (i < pv.lmax - m * pv.mres + 1) return pv.ab[col_ext(pv, m, 0) + i];
    if (i == 1) return make_double2(sqrt(2.0 * dm + 3.0), 0.0);
    return make_double2(sqrt((4.0 * n * n - 1.0) / (n * n - dm * dm)),
                        -sqrt((2.0 * n + 1.0) / (2.0 * n - 3.0) * (n1 * n1 - dm * dm) / (n * n - dm * dm)));
}
__device__ double plain_eps(const PlanView<double> &pv, int m, int i)
{
    const double dm = m * pv.mres, n = dm + i;
    return i == 0 ? 0.0 : sqrt((n * n - dm * dm) / (4.0 * n * n - 1.0));
}

// A vector transform whose plan has no tables -- a first call that is captured, in
// which nothing can be allocated, or tables that do not fit -- computes them as it
// goes: (a_n, b_n), eps_n and the segments' states, stepped to from P_m^m.  The
// same values bit for bit, at the cost of the steps (a segment in the middle of an
// order of 32 S degrees takes 16 S of them).  The kernels' parameter TAB.
__device__ __forceinline__ double eps_at(const PlanView<double> &pv, long colx, int m, int i)
{
    return pv.eps ? pv.eps[colx + i] : plain_eps(pv, m, i);
}

// One step of the recurrence, y_n = a x y_{n-1} + b y_{n-2}, and the factor s_n of
// the value, at degree m mres + i: (beta_n, s_n) of Q_n, where a = 1 is left out by
// the caller, or (a_n, b_n) of P_n itself (`plain`).  Zeros past the order's last degree.
// col: the order's first index in the tables.
struct Step { double a, b, s; };
template <bool TAB>
__device__ __forceinline__ Step step_of(const PlanView<double> &pv, long col, int m, int i, bool in, bool plain)
{
    Step r = {0.0, 0.0, 0.0};
    if (!in) return r;
    const double2 v = TAB ? __ldg((plain ? pv.abx : pv.qs) + col + i) : plain_ab(pv, m, i);
    if (plain) {
        r.a = v.x;
        r.b = v.y;
        r.s = 1.0;
    } else {
        r.b = v.x;
        r.s = v.y;
    }
    return r;
}

// The state entering a segment for pair p, y 2^(-240 k): of Q, or of P (`plain`).
struct State { double y1, y2; int k; };
__device__ State stepped_state(const PlanView<double> &pv, int m, int seg, int p)
{
    const double x = pv.x[p];
    State v = {0.0, pv.pmm[(size_t)m * pv.npairs + p], pv.pmmk[(size_t)m * pv.npairs + p]};
    const double2 *ab = pv.ab + col_ext(pv, m, 0);
    for (int i = 0; i < seg * kSeedSeg; ++i) {   // as k_build_restarts
        const double yn = fma(ab[i].x * x, v.y1, ab[i].y * v.y2);
        v.y2 = v.y1;
        v.y1 = yn;
        if (v.k > 0 && (__double2hiint(yn) & 0x7fffffff) >= kHiOne) {
            v.y1 *= kDown;
            v.y2 *= kDown;
            v.k -= 1;
        }
    }
    return v;
}
template <bool TAB>
__device__ __forceinline__ State state_of(const PlanView<double> &pv, int m, int seg, int p, bool plain)
{
    if (!TAB) return stepped_state(pv, m, seg, p);
    const size_t i = pv.segoff[m] + seg, o = i * pv.npairs + p;
    const double2 v = __ldg(pv.seeds64 + o);
    // the power of two that takes the segment's stored state back to P
    const double down = plain ? __hiloint2double((1023 - __ldg(pv.hseg + i)) << 20, 0) : 1.0;
    return State{v.x * down, v.y * down, __ldg(pv.seeds64k + o)};
}

// |Q| s >= 1 to within the 2^-20 of the high words' sum (a rescaling test: see
// Sec. 3.5; hs = high word of s less that of 1).
__device__ __forceinline__ bool reaches_one(double q, int hs)
{
    return (__double2hiint(q) & 0x7fffffff) + hs >= kHiOne;
}

// ---------------------------------------------------------------------------
// Scalar synthesis.  A CTA of four warps (one per SM quarter) per (order m, 32
// latitude pairs, BC fields).  It takes the degrees four segments at a time: each
// warp generates P of one segment, one pair per lane, and the segment's spectral
// values times s_n into shared memory; then warp w sums the pairs 8 w .. 8 w + 7,
// lane (pairs, parity, c) the products of component c (field, real/imaginary) over
// the degrees of one parity of n - m.  With C = 2 BC components 16 / C lanes share
// the 8 pairs of a component and parity (16 fields: a lane takes both parities).
// Every sum runs over the degrees in order whatever BC is, so a field's result
// does not depend on the batch it comes in (lanes as slices of the degrees took
// the same time).  The sums are spread evenly over the SM quarters whatever the
// number of segments (2 x 16 vector fields at N = 127: 165 us with a warp per
// segment and 16 fields, 130 us).  16 fields at N = 511: 1981 us with three
// instructions per step and 8 fields, 1766 with two and 16 fields a warp, 1653 us;
// one field at N = 255: 134 -> 42 us.  vec: the spectra run to degree lmax + 1,
// the recurrence is Sec. 3.2's, and the sums are divided by sin(theta).
// ---------------------------------------------------------------------------
constexpr int kSynWarps = 4;
// row of the P tile: 32 pairs, 16-byte aligned rows on shifted banks (two rows by four
// lanes of one pair each at 1 field)
template <int BC> constexpr int kSynRow = BC == 1 ? 36 : 34;
template <int BC> constexpr size_t synth64_smem()
{
    return sizeof(double) * (kSynWarps * kSeedSeg * ((2 * BC + 2) + kSynRow<BC>));
}

template <int BC, bool TAB>
__global__ void __launch_bounds__(32 * kSynWarps)
k_synth64(PlanView<double> pv, const double *__restrict__ spec, VecSpec vs, double *__restrict__ eo, int batch,
          int ngroups, int nchunk, int nsm, int vec, int op)
{
    // PW pairs per warp; a lane takes NP of them and PAR parities
    constexpr int C = 2 * BC, W = kSynWarps, FS = C + 2, PW = 32 / W, PAR = C == 32 ? 2 : 1, NP = C == 32 ? PW : PW * C / 16;
    constexpr int kRow = kSynRow<BC>;
    extern __shared__ __align__(16) double s_mem[];
    double *s_f = s_mem;                              // [W kSeedSeg degrees][FS]
    double *s_P = s_mem + W * kSeedSeg * FS;          // [W kSeedSeg degrees][kRow]
    __shared__ double s_a[W][kMaxDeg], s_beta[W][kMaxDeg];
    __shared__ int s_hs[W][kMaxDeg];

    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int item = snake(blockIdx.x, gridDim.x, nsm);
    const int chunk = item % nchunk, rest = item / nchunk;
    const int g = rest % ngroups, m = rest / ngroups;
    const int b0 = chunk * BC;
    const int npairs = pv.npairs, Ls = pv.lmax - m * pv.mres + 1, L = Ls + vec;
    const int nseg = (Ls + kSeedSeg - 1) / kSeedSeg, ntask = (L + kSeedSeg - 1) / kSeedSeg;
    const long colq = col_ext(pv, m, 1), col = col_ext(pv, m, 0);
    const double2 *spec2 = reinterpret_cast<const double2 *>(spec);
    const int p = g * 32 + lane;
    const bool valid = p < npairs;
    const double x = valid ? pv.x[p] : 0.0;
    const int first = TAB ? (vec ? pv.glive_vec : pv.glive)[(size_t)m * ngroups + g] : 0;
    const double insc = (op == OP_ANALYS_ADJ && m > 0) ? 0.5 : 1.0;   // adjoint of analysis: b / c_m
    const int c = lane % C, par = PAR == 2 ? 0 : (lane / C) & 1, pq = PW * w + (PAR == 2 ? 0 : lane / (2 * C)) * NP;
    const int u = (w + item) & (W - 1);   // the segment of a block this warp generates (turned from CTA to CTA)

    double acc[PAR][NP];
#pragma unroll
    for (int q = 0; q < NP; ++q)
#pragma unroll
        for (int r = 0; r < PAR; ++r) acc[r][q] = 0.0;

    for (int sb = first; sb < ntask; sb += W) {
        const int sg = sb + u;
        if (sg < ntask) {
            // `vec`: the degree lmax + 1 is a segment of its own when the order's
            // degrees fill theirs; it continues the last one's recurrence
            const bool tail = sg == nseg;
            const int seg = tail ? nseg - 1 : sg;
            const int cnt = min(kSeedSeg, L - sg * kSeedSeg);
            const int nstep = tail ? kSeedSeg + 1 : (cnt + 15) & ~15;
            double y1 = 0.0, y2 = 0.0;
            int k = 0;
            if (valid) {
                const State v = state_of<TAB>(pv, m, seg, p, vec);
                y1 = v.y1;
                y2 = v.y2;
                k = v.k;
            }
            double fs = 1.0;   // s_n of this lane's degree
            for (int t = lane; t < nstep; t += 32) {
                const int d = seg * kSeedSeg + t;
                const Step st = step_of<TAB>(pv, colq, m, d, d < L, vec);
                s_a[u][t] = st.a;
                s_beta[u][t] = st.b;
                s_hs[u][t] = __double2hiint(st.s) - kHiOne;
                if (t < kSeedSeg) fs = st.s;
            }
            const double sc = vec ? 1.0 : fs * insc;
            double *row = s_f + (u * kSeedSeg + lane) * FS;
            // this lane's degree of field f: at (f < nb ? pa : pb) + f * step
            const int i = sg * kSeedSeg + lane;
            const bool top = i == Ls;
            const int nb = vec ? vs.nb : batch;
            const size_t step = top ? pv.mmax + 1 : pv.nlm;
            const double2 *pa = top ? vs.top + m : (vec ? vs.u : spec2) + col + i;
            const double2 *pb = top ? pa : vs.w + col + i - (size_t)nb * pv.nlm;
#pragma unroll
            for (int b = 0; b < BC; ++b) {
                double2 f = make_double2(0.0, 0.0);
                if (lane < cnt && b0 + b < batch) {
                    f = __ldg((b0 + b < nb ? pa : pb) + (size_t)(b0 + b) * step);
                    if (!vec) {
                        f.x *= sc;
                        f.y *= sc;
                    }
                    if (m == 0) f.y = 0.0;
                }
                *reinterpret_cast<double2 *>(row + 2 * b) = f;
            }
            __syncwarp();
            double *Pt = s_P + u * kSeedSeg * kRow + lane;
            const bool scaled = __any_sync(kFull, k > 0);
            for (int t = 0; t < nstep; ++t) {
                double yn = fma(vec ? s_a[u][t] * x : x, y1, s_beta[u][t] * y2);
                y2 = y1;
                double v = yn;
                if (scaled) {   // some pair still carries a scaled value (Sec. 3.5)
                    if (k > 0 && reaches_one(yn, s_hs[u][t])) {
                        yn *= kDown;
                        y2 *= kDown;
                        k -= 1;
                    }
                    v = k == 0 ? yn : 0.0;
                }
                y1 = yn;
                if (!tail) Pt[t * kRow] = v;
                else if (t == kSeedSeg) Pt[0] = v;
                else if (t > 0 && t < 16) Pt[t * kRow] = 0.0;
            }
        }
        __syncthreads();
        // rows past the order's last degree, up to a multiple of 16, hold zeros times finite values
        const int nd = min(W * kSeedSeg, L - sb * kSeedSeg);
        const double *fd = s_f + par * FS + c, *Pd = s_P + par * kRow + pq;
        const int nj = (nd + 1) / 2;
#pragma unroll (NP >= 8 ? 2 : 16 / NP)
        for (int j = 0; j < nj; ++j) {
#pragma unroll
            for (int r = 0; r < PAR; ++r) {
                const double f = fd[(2 * j + r) * FS];
                const double *Pj = Pd + (2 * j + r) * kRow;
                if constexpr (NP == 1) {
                    acc[r][0] = fma(f, Pj[0], acc[r][0]);
                } else {
#pragma unroll
                    for (int q = 0; q < NP / 2; ++q) {
                        const double2 v = reinterpret_cast<const double2 *>(Pj)[q];
                        acc[r][2 * q] = fma(f, v.x, acc[r][2 * q]);
                        acc[r][2 * q + 1] = fma(f, v.y, acc[r][2 * q + 1]);
                    }
                }
            }
        }
        __syncthreads();
    }
    // [field][pair][E, O][part], in the P tile
#pragma unroll
    for (int r = 0; r < PAR; ++r)
#pragma unroll
        for (int q = 0; q < NP; ++q) s_P[(((c >> 1) * 32 + pq + q) * 2 + par + r) * 2 + (c & 1)] = acc[r][q];
    __syncthreads();
    double2 *eo2 = reinterpret_cast<double2 *>(eo);
    for (int i = threadIdx.x; i < BC * 64; i += 32 * W) {
        const int b = i >> 6, q = g * 32 + ((i & 63) >> 1);
        if (b0 + b >= batch || q >= npairs) continue;
        double2 v = reinterpret_cast<const double2 *>(s_P)[i];
        if (vec) {
            const double is = 1.0 / pv.st[q];
            v.x *= is;
            v.y *= is;
        }
        eo2[(((size_t)vs.inter(b0 + b) * (pv.mmax + 1) + m) * npairs + q) * 2 + (i & 1)] = v;
    }
}

// ---------------------------------------------------------------------------
// Scalar analysis.  A CTA of four warps (one per SM quarter) per (order m,
// segment of kSeedSeg degrees, BC fields).  It takes the latitude pairs 128 at a
// time: each warp generates P of the segment for 32 of them, one pair per lane,
// into shared memory; then warp w sums degrees 8 w .. 8 w + 7 over all 128,
// lane (degrees, half, c) the products of component c (field, real/imaginary) over
// the even or the odd pairs.  With C = 2 BC components 16 / C lanes share the 8
// degrees of a component and half (16 fields: a lane takes both halves), and the
// sum over latitudes needs one exchange per degree; a lane per pair instead needs
// an FP64 butterfly over all 32 lanes for every 16 / BC degrees -- with 96 pairs a
// third on top of the sums -- and a warp per segment leaves SM quarters idle where
// segments are few.  Every half is summed over its pairs in order whatever BC is,
// so a field's result does not depend on the batch it comes in.  16 fields at
// N = 511: 2357 us with lanes as pairs and 8 fields, 1644 us (1636 with lanes as
// slices of the pairs, 32 / C of them, whose sums depended on BC); 2 x 16 vector
// fields at N = 127: 926 -> 164 us; one field at N = 255: 67 -> 43 us.  The groups
// of 32 pairs before the first one with a live pair in the segment (static polar
// optimisation, Sec. 3.1) are left out.
//
// blockIdx: x segment (with `vec`, see k_synth64, the degree lmax + 1 is one
// more, alone in its block when the order's degrees fill their segments: it
// continues the recurrence of the last segment), y order index, z field chunk.
// ---------------------------------------------------------------------------
constexpr int kAnaWarps = 4;

template <int BC, bool TAB>
__global__ void __launch_bounds__(32 * kAnaWarps)
k_analys64(PlanView<double> pv, const double *__restrict__ sd, double *__restrict__ spec, VecSpec vs, int batch,
           int vec, int op)
{
    // DB degrees per warp; a lane takes ND of them and HV halves of the pairs (the even, the odd ones)
    constexpr int C = 2 * BC, W = kAnaWarps, DB = kSeedSeg / W, HV = C == 32 ? 2 : 1, ND = C == 32 ? DB : DB * C / 16;
    // folds in flight: pairs of a half ahead of the sums, one fold per pair where a lane has one degree
    constexpr int AH = 16 / ND / HV, NF = ND == 1 ? 1 : 2;
    __shared__ double s_P[W][kSeedSeg][33];
    __shared__ double s_a[kSeedSeg + DB], s_beta[kSeedSeg + DB];
    __shared__ int s_hs[kSeedSeg + DB];
    __shared__ int s_g0;

    const int m = blockIdx.y, b0 = blockIdx.z * BC, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int npairs = pv.npairs, ngroups = (npairs + 31) >> 5;
    const int Ls = pv.lmax - m * pv.mres + 1, L = Ls + vec;
    const int nseg = (Ls + kSeedSeg - 1) / kSeedSeg;
    const bool tail = (int)blockIdx.x == nseg;   // the degree lmax + 1 alone
    const int seg = tail ? nseg - 1 : blockIdx.x;
    const int n0 = blockIdx.x * kSeedSeg;        // first degree summed
    if (n0 >= L) return;
    const int cnt = min(kSeedSeg, L - n0);
    const int nstep = tail ? kSeedSeg + 1 : (cnt + DB - 1) & ~(DB - 1);
    const long colq = col_ext(pv, m, 1) + seg * kSeedSeg, col = col_ext(pv, m, 0) + n0;
    if (threadIdx.x == 0) s_g0 = ngroups;
    if (threadIdx.x < nstep) {
        const int t = threadIdx.x;
        const Step st = step_of<TAB>(pv, colq - seg * kSeedSeg, m, seg * kSeedSeg + t, seg * kSeedSeg + t < L, vec);
        s_a[t] = st.a;
        s_beta[t] = st.b;
        s_hs[t] = __double2hiint(st.s) - kHiOne;
    }
    if (tail)   // one degree: the rest of its block of DB is zero
        for (int t = 1; t < DB; ++t) s_P[w][t][lane] = 0.0;
    __syncthreads();
    for (int g = threadIdx.x; g < ngroups; g += 32 * W)
        if (!TAB || (vec ? pv.glive_vec : pv.glive)[(size_t)m * ngroups + g] <= seg) {
            atomicMin(&s_g0, g);
            break;
        }
    __syncthreads();
    const int g0 = s_g0;

    // this lane's component, half and degrees
    const int c = lane % C, half = HV == 2 ? 0 : (lane / C) & 1, b = b0 + (c >> 1);
    const int dw = w * DB, d0 = dw + (HV == 2 ? 0 : lane / (2 * C)) * ND;
    // s at 4 q, d at 4 q + 2 (a lane with one degree: the one its parity takes)
    const double *fold = sd + ((size_t)vs.inter(b) * (pv.mmax + 1) + m) * npairs * 4 + (c & 1) + (ND == 1 ? 2 * (d0 & 1) : 0);
    const bool has = b < batch && dw < cnt;
    double acc[HV][ND];
#pragma unroll
    for (int h = 0; h < HV; ++h)
#pragma unroll
        for (int t = 0; t < ND; ++t) acc[h][t] = 0.0;

    for (int gb = g0; gb < ngroups; gb += W) {
        const int p = (gb + w) * 32 + lane;
        const bool valid = p < npairs;
        double x = 0.0, y1 = 0.0, y2 = 0.0;
        int k = 0;
        if (valid) {
            const State v = state_of<TAB>(pv, m, seg, p, vec);
            x = pv.x[p];
            y1 = v.y1;
            y2 = v.y2;
            k = v.k;
        }
        // the folds, AH pairs of a half ahead of the sums
        const int nq = min(64, (npairs - gb * 32 + 1) / 2);   // pairs of a half in this block
        double fv[AH][HV][NF];
        const auto fetch = [&](int j, int h, double (&f)[NF]) {
            const int q = gb * 32 + 2 * j + half + h;
            const bool in = has && j < nq && q < npairs;
#pragma unroll
            for (int i = 0; i < NF; ++i) f[i] = in ? __ldg(fold + (size_t)q * 4 + 2 * i) : 0.0;
        };
#pragma unroll
        for (int u = 0; u < AH; ++u)
#pragma unroll
            for (int h = 0; h < HV; ++h) fetch(u, h, fv[u][h]);
        __syncthreads();   // the last block's sums are done with s_P
        if (gb + w < ngroups) {
            const bool scaled = __any_sync(kFull, k > 0);
            for (int t = 0; t < nstep; ++t) {
                double yn = fma(vec ? s_a[t] * x : x, y1, s_beta[t] * y2);
                y2 = y1;
                double v = yn;
                if (scaled) {   // some pair still carries a scaled value (Sec. 3.5)
                    if (k > 0 && reaches_one(yn, s_hs[t])) {
                        yn *= kDown;
                        y2 *= kDown;
                        k -= 1;
                    }
                    v = k == 0 ? yn : 0.0;
                }
                y1 = yn;
                if (!tail) s_P[w][t][lane] = v;
                else if (t == kSeedSeg) s_P[w][0][lane] = v;
            }
        }
        __syncthreads();
        if (dw < cnt) {
            const auto add = [&](int j, double (&f)[HV][NF]) {
#pragma unroll
                for (int h = 0; h < HV; ++h) {
                    const int r = 2 * j + half + h;   // pair within the block
                    const double *P = &s_P[r >> 5][d0][r & 31];
                    const double s = f[h][0], d = f[h][NF - 1];
                    if (ND == DB) fetch(j + AH, h, f[h]);   // (few pairs ahead: before the sums)
#pragma unroll
                    for (int t = 0; t < ND; ++t) acc[h][t] = fma(P[t * 33], (t & 1) ? d : s, acc[h][t]);
                    if (ND < DB) fetch(j + AH, h, f[h]);
                }
            };
            int j = 0;
#pragma unroll 1
            for (; j + AH <= nq; j += AH)
#pragma unroll
                for (int u = 0; u < AH; ++u) add(j + u, fv[u]);
#pragma unroll
            for (int u = 0; u < AH - 1; ++u)
                if (j + u < nq) add(j + u, fv[u]);
        }
    }
    // even and odd pairs
#pragma unroll
    for (int t = 0; t < ND; ++t) acc[0][t] += HV == 2 ? acc[HV - 1][t] : __shfl_xor_sync(kFull, acc[0][t], C & 31);
    __syncthreads();
#pragma unroll
    for (int t = 0; t < ND; ++t) s_P[0][d0 + t][c] = acc[0][t];   // the same from either half's lane
    __syncthreads();
    if (lane >= cnt) return;
    // P_n = s_n Q_n; c_m for the adjoint of synthesis
    const double sc = (vec ? 1.0 : __ldg(&pv.qs[colq + lane].y)) * ((op == OP_SYNTH_ADJ && m > 0) ? 2.0 : 1.0);
    double2 *spec2 = reinterpret_cast<double2 *>(spec);
    for (int i = w; i < BC && b0 + i < batch; i += W) {
        double2 *dst = vec ? vs.field(b0 + i, pv.nlm) : spec2 + (size_t)(b0 + i) * pv.nlm;
        dst = n0 + lane < Ls ? dst + col + lane : vs.top + (size_t)(b0 + i) * (pv.mmax + 1) + m;
        *dst = make_double2(s_P[0][lane][2 * i] * sc, m == 0 ? 0.0 : s_P[0][lane][2 * i + 1] * sc);
    }
}

// ---------------------------------------------------------------------------
// Vector transforms: spectra in and out of the scalar sums (see the head of
// this file).  U and W (degrees to lmax) are written where the grids will be,
// which the FFT fills last: nlm <= nlat nphi / 2.  A and B come in the place of S
// and T.  Only the degree lmax + 1 needs room of its own (VecSpec::top).
// ---------------------------------------------------------------------------
// Thread per (degree, order index m = blockIdx.y, field blockIdx.z).
__global__ void __launch_bounds__(128)
k_vec64_split(PlanView<double> pv, const double2 *__restrict__ S, const double2 *__restrict__ T, VecSpec vs, int op)
{
    const int m = blockIdx.y, b = blockIdx.z, dm = m * pv.mres;
    const int L = pv.lmax - dm + 1;
    const int i = blockIdx.x * blockDim.x + threadIdx.x;   // degree k = dm + i, up to lmax + 1
    if (i > L) return;
    const long col = col_ext(pv, m, 0), colx = col_ext(pv, m, 1);
    const double2 *Sb = S + (size_t)b * pv.nlm + col, *Tb = T + (size_t)b * pv.nlm + col;
    const double k = dm + i;
    // adjoint of analysis: b / (c_m n (n + 1)), nothing at n = 0
    const auto load = [&](const double2 *a, int j) {
        if (j < 0 || j >= L) return make_double2(0.0, 0.0);
        double2 v = a[j];
        if (m == 0) v.y = 0.0;
        if (op == OP_ANALYS_ADJ) {
            const double n = dm + j, sc = n == 0.0 ? 0.0 : (m > 0 ? 0.5 : 1.0) / (n * (n + 1.0));
            v.x *= sc;
            v.y *= sc;
        }
        return v;
    };
    const double lo = (k - 1.0) * eps_at(pv, colx, m, i), hi = i < L ? (k + 2.0) * eps_at(pv, colx, m, i + 1) : 0.0;
    const double2 Sl = load(Sb, i - 1), Sc = load(Sb, i), Sh = load(Sb, i + 1);
    const double2 Tl = load(Tb, i - 1), Tc = load(Tb, i), Th = load(Tb, i + 1);
    double2 U, W;
    U.x = lo * Sl.x - hi * Sh.x + dm * Tc.y;
    U.y = lo * Sl.y - hi * Sh.y - dm * Tc.x;
    W.x = lo * Tl.x - hi * Th.x - dm * Sc.y;
    W.y = lo * Tl.y - hi * Th.y + dm * Sc.x;
    if (i < L) {
        vs.u[(size_t)b * pv.nlm + col + i] = U;
        vs.w[(size_t)b * pv.nlm + col + i] = W;
    } else {
        vs.top[(size_t)b * (pv.mmax + 1) + m] = U;
        vs.top[(size_t)(vs.nb + b) * (pv.mmax + 1) + m] = W;
    }
}

// In place; a CTA per (order index m = blockIdx.x, field blockIdx.y) takes the degrees
// blockDim.x at a time, each block's values read before any is overwritten, and the
// last of a block handed on to the next.
__global__ void __launch_bounds__(128) k_vec64_join(PlanView<double> pv, VecSpec vs, int op)
{
    __shared__ double2 s_last[2][2];   // A and B of the degree before the block, of this and the next
    const int m = blockIdx.x, b = blockIdx.y, dm = m * pv.mres;
    const int L = pv.lmax - dm + 1;
    const long col = col_ext(pv, m, 0), colx = col_ext(pv, m, 1);
    double2 *A = vs.u + (size_t)b * pv.nlm + col, *B = vs.w + (size_t)b * pv.nlm + col;
    const double2 At = vs.top[(size_t)b * (pv.mmax + 1) + m], Bt = vs.top[(size_t)(vs.nb + b) * (pv.mmax + 1) + m];
    const double2 z = make_double2(0.0, 0.0);
    if (threadIdx.x < 2) s_last[0][threadIdx.x] = z;
    __syncthreads();
    for (int i0 = 0, q = 0; i0 < L; i0 += blockDim.x, q ^= 1) {
        const int i = i0 + threadIdx.x;   // degree n = dm + i
        const bool in = i < L;
        double2 Al = z, Ac = z, Ah = z, Bl = z, Bc = z, Bh = z;
        if (in) {
            Ac = A[i];
            Bc = B[i];
            Ah = i + 1 < L ? A[i + 1] : At;
            Bh = i + 1 < L ? B[i + 1] : Bt;
            Al = threadIdx.x > 0 ? A[i - 1] : s_last[q][0];
            Bl = threadIdx.x > 0 ? B[i - 1] : s_last[q][1];
        }
        if (threadIdx.x == blockDim.x - 1) {
            s_last[q ^ 1][0] = Ac;
            s_last[q ^ 1][1] = Bc;
        }
        __syncthreads();
        if (!in) continue;
        const double n = dm + i;
        const double hi = n * eps_at(pv, colx, m, i + 1), lo = i > 0 ? (n + 1.0) * eps_at(pv, colx, m, i) : 0.0;
        double sc;
        if (op == OP_SYNTH_ADJ) sc = m > 0 ? 2.0 : 1.0;
        else sc = n == 0.0 ? 0.0 : 1.0 / (n * (n + 1.0));
        double2 s, t;
        s.x = sc * (hi * Ah.x - lo * Al.x + dm * Bc.y);
        s.y = sc * (hi * Ah.y - lo * Al.y - dm * Bc.x);
        t.x = sc * (hi * Bh.x - lo * Bl.x - dm * Ac.y);
        t.y = sc * (hi * Bh.y - lo * Bl.y + dm * Ac.x);
        if (m == 0) s.y = t.y = 0.0;
        A[i] = s;
        B[i] = t;
    }
}

// ---------------------------------------------------------------------------
// Plan tables: (beta_n, s_n), (a_n, b_n) and eps_n of every degree m .. lmax + 1
// of every order, and per segment the exponent h of its states' scale.  s_n^2 is
// the product of (4 j^2 - 1) / (j^2 - m^2) over the segment, formed in
// double-double arithmetic (Dekker 1971).  A warp per (segment, order index
// blockIdx.y), a degree per lane, the product by a scan (a thread per segment
// took 100 us of divisions and roots one after the other).
// ---------------------------------------------------------------------------
struct dd { double h, l; };
__device__ __forceinline__ dd dd_norm(double h, double l)
{
    dd r;
    r.h = h + l;
    r.l = l - (r.h - h);
    return r;
}
__device__ __forceinline__ dd dd_mul(dd a, dd b)
{
    const double p = a.h * b.h;
    return dd_norm(p, fma(a.l, b.h, fma(a.h, b.l, fma(a.h, b.h, -p))));
}

__global__ void __launch_bounds__(32)
k_build_qs(PlanView<double> pv, const unsigned long long *__restrict__ segoff, double2 *__restrict__ qs,
           double2 *__restrict__ abx, double *__restrict__ eps, int *__restrict__ hseg)
{
    const int m = blockIdx.y, seg = blockIdx.x, lane = threadIdx.x;
    const double dm = m * pv.mres;
    const int Ls = pv.lmax - m * pv.mres + 1;
    const int nseg = (Ls + kSeedSeg - 1) / kSeedSeg;
    if (seg >= nseg) return;
    const long colx = col_ext(pv, m, 1);
    const int i0 = seg * kSeedSeg;
    const auto ratio = [&](int i) {   // s_n^2 / s_{n-1}^2 at degree dm + i
        dd r = {1.0, 0.0};
        if (i == 0) return r;
        const double n = dm + i, num = 4.0 * n * n - 1.0, den = n * n - dm * dm;   // exact
        const double q = num / den;
        return dd_norm(q, fma(-q, den, num) / den);
    };
    const auto put = [&](int i, dd s2, int h) {
        const double n = dm + i, n1 = n - 1.0;
        if (i == 0) {   // Q_m is the start value P_m^m, handed over as Q_{m-2}
            qs[colx] = make_double2(1.0, scalbn(1.0, -h));
            abx[colx] = plain_ab(pv, m, 0);
            eps[colx] = 0.0;
            return;
        }
        const double bb = i == 1 ? 0.0 : (n1 * n1 - dm * dm) / (4.0 * n1 * n1 - 1.0);   // eps_{n-1}^2
        qs[colx + i] = make_double2(i == i0 ? -sqrt(bb) : -bb, scalbn(sqrt(s2.h), -h));
        eps[colx + i] = plain_eps(pv, m, i);
        abx[colx + i] = plain_ab(pv, m, i);
    };
    dd s2 = ratio(i0 + lane);
#pragma unroll
    for (int o = 1; o < 32; o *= 2) {
        dd u;
        u.h = __shfl_up_sync(kFull, s2.h, o);
        u.l = __shfl_up_sync(kFull, s2.l, o);
        if (lane >= o) s2 = dd_mul(s2, u);
    }
    // half of the growth of s over the segment's degrees
    const int h = __shfl_sync(kFull, ilogb(s2.h) / 4, min(kSeedSeg, Ls - i0) - 1);
    if (lane == 0) hseg[segoff[m] + seg] = h;
    if (i0 + lane <= Ls) put(i0 + lane, s2, h);
    if (lane == kSeedSeg - 1 && i0 + kSeedSeg == Ls) put(Ls, dd_mul(s2, ratio(Ls)), h);
}

// Fields per CTA {1, 2, 4, 8, 16}: the width with the shortest busiest SM -- CTAs
// per SM, rounded up, times the FP64 instructions of one (2 per degree and 32
// pairs to generate P, 2 per field to sum).
inline int pick_width(long units, int batch)
{
    const long sms = sm_count();
    long best = 0;
    int bc = 1;
    for (int f = 16; f >= 1; f /= 2) {
        const long ctas = units * ((batch + f - 1) / f);
        const long t = (ctas + sms - 1) / sms * (1 + f);
        if (best == 0 || t < best) {
            best = t;
            bc = f;
        }
    }
    return bc;
}

// All of the tables, or with `vec` none of them.
bool tables_ok(const PlanView<double> &pv, bool vec)
{
    if (vec && !pv.seeds64) return pv.ab && pv.pmm && pv.pmmk && !pv.eps;
    return pv.segoff && pv.seeds64 && pv.seeds64k && pv.glive && pv.glive_vec && pv.qs && pv.abx && pv.eps && pv.hseg;
}

template <int BC, bool TAB = true>
cudaError_t synth64_go(const PlanView<double> &pv, const double *spec, const VecSpec *vs, double *eo, int batch, Op op,
                       cudaStream_t s)
{
    const int ng = (pv.npairs + 31) / 32, nc = (batch + BC - 1) / BC;
    constexpr size_t smem = synth64_smem<BC>();
    if (smem > 40 * 1024) {
        cudaError_t e = cudaFuncSetAttribute(k_synth64<BC, TAB>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        if (e != cudaSuccess) return e;
    }
    const long items = (long)(pv.mmax + 1) * ng * nc;
    k_synth64<BC, TAB><<<(unsigned)items, 32 * kSynWarps, smem, s>>>(pv, spec, vs ? *vs : VecSpec(), eo, batch, ng, nc,
                                                                sm_count(), vs ? 1 : 0, (int)op);
    return cudaGetLastError();
}

// Scalar from `spec`, or with `vs` the scalar form of a vector transform, from its spectra.
cudaError_t synth64(const PlanView<double> &pv, const double *spec, const VecSpec *vs, double *eo, int batch, Op op,
                    int bc, cudaStream_t s)
{
    if (!tables_ok(pv, vs != nullptr)) return cudaErrorInvalidValue;
    if (!pv.seeds64) return synth64_go<8, false>(pv, spec, vs, eo, batch, op, s);
    if (bc <= 0) bc = pick_width((long)(pv.mmax + 1) * ((pv.npairs + 31) / 32), batch);
    switch (bc) {
    case 1: return synth64_go<1>(pv, spec, vs, eo, batch, op, s);
    case 2: return synth64_go<2>(pv, spec, vs, eo, batch, op, s);
    case 4: return synth64_go<4>(pv, spec, vs, eo, batch, op, s);
    case 8: return synth64_go<8>(pv, spec, vs, eo, batch, op, s);
    case 16: return synth64_go<16>(pv, spec, vs, eo, batch, op, s);
    default: return cudaErrorInvalidValue;
    }
}

template <int BC, bool TAB = true>
cudaError_t analys64_go(const PlanView<double> &pv, const double *sd, double *spec, const VecSpec *vs, int batch,
                        Op op, cudaStream_t s)
{
    const dim3 grid((unsigned)((pv.lmax + (vs ? 1 : 0) + kSeedSeg) / kSeedSeg), (unsigned)(pv.mmax + 1),
                    (unsigned)((batch + BC - 1) / BC));
    k_analys64<BC, TAB><<<grid, 32 * kAnaWarps, 0, s>>>(pv, sd, spec, vs ? *vs : VecSpec(), batch, vs ? 1 : 0, (int)op);
    return cudaGetLastError();
}

// Segments of all orders (orders k mres, degrees k mres .. lmax).
inline long segments(const PlanView<double> &pv)
{
    long n = 0;
    for (int k = 0; k <= pv.mmax; ++k) n += (pv.lmax - k * pv.mres + kSeedSeg) / kSeedSeg;
    return n;
}

cudaError_t analys64(const PlanView<double> &pv, const double *sd, double *spec, const VecSpec *vs, int batch, Op op,
                     int bc, cudaStream_t s)
{
    if (!tables_ok(pv, vs != nullptr)) return cudaErrorInvalidValue;
    if (!pv.seeds64) return analys64_go<8, false>(pv, sd, spec, vs, batch, op, s);
    if (bc <= 0) bc = pick_width(segments(pv), batch);
    switch (bc) {
    case 1: return analys64_go<1>(pv, sd, spec, vs, batch, op, s);
    case 2: return analys64_go<2>(pv, sd, spec, vs, batch, op, s);
    case 4: return analys64_go<4>(pv, sd, spec, vs, batch, op, s);
    case 8: return analys64_go<8>(pv, sd, spec, vs, batch, op, s);
    case 16: return analys64_go<16>(pv, sd, spec, vs, batch, op, s);
    default: return cudaErrorInvalidValue;
    }
}

}  // namespace

cudaError_t launch_build_qs(const PlanView<double> &pv, const unsigned long long *segoff, double2 *qs, double2 *abx,
                            double *eps, int *hseg, cudaStream_t st)
{
    const int nseg = (pv.lmax + kSeedSeg) / kSeedSeg;
    k_build_qs<<<dim3((unsigned)nseg, (unsigned)(pv.mmax + 1)), 32, 0, st>>>(pv, segoff, qs, abx, eps, hseg);
    return cudaGetLastError();
}

cudaError_t launch_synth64(const PlanView<double> &pv, const double *spec, double *eo, int batch, Op op, int bc,
                           cudaStream_t s)
{
    return synth64(pv, spec, nullptr, eo, batch, op, bc, s);
}

cudaError_t launch_analys64(const PlanView<double> &pv, const double *sd, double *spec, int batch, Op op, int bc,
                            cudaStream_t s)
{
    return analys64(pv, sd, spec, nullptr, batch, op, bc, s);
}

cudaError_t launch_synth_vec64(const PlanView<double> &pv, const double *S, const double *Tc, double *vt, double *vp,
                               double2 *top, double *eo, int batch, Op op, cudaStream_t s)
{
    if (!tables_ok(pv, true)) return cudaErrorInvalidValue;
    const size_t ngrid = (size_t)pv.nlat * pv.nphi, nspec = (size_t)pv.nlm * 2;
    cudaError_t e = cudaSuccess;
    for (int b0 = 0; b0 < batch && e == cudaSuccess; b0 += kVec64Group) {
        const int nb = batch - b0 < kVec64Group ? batch - b0 : kVec64Group;
        const VecSpec vs = {reinterpret_cast<double2 *>(vt + b0 * ngrid), reinterpret_cast<double2 *>(vp + b0 * ngrid),
                            top, nb, b0, batch + b0 - nb};
        const dim3 grid((unsigned)((pv.lmax + 2 + 127) / 128), (unsigned)(pv.mmax + 1), (unsigned)nb);
        k_vec64_split<<<grid, 128, 0, s>>>(pv, reinterpret_cast<const double2 *>(S + b0 * nspec),
                                           reinterpret_cast<const double2 *>(Tc + b0 * nspec), vs, (int)op);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = synth64(pv, nullptr, &vs, eo, 2 * nb, OP_SYNTH, 0, s);
    }
    return e;
}

cudaError_t launch_analys_vec64(const PlanView<double> &pv, const double *sd, double2 *top, double *S, double *Tc,
                                int batch, Op op, cudaStream_t s)
{
    const size_t nspec = (size_t)pv.nlm * 2;
    cudaError_t e = cudaSuccess;
    for (int b0 = 0; b0 < batch && e == cudaSuccess; b0 += kVec64Group) {
        const int nb = batch - b0 < kVec64Group ? batch - b0 : kVec64Group;
        const VecSpec vs = {reinterpret_cast<double2 *>(S + b0 * nspec), reinterpret_cast<double2 *>(Tc + b0 * nspec),
                            top, nb, b0, batch + b0 - nb};
        e = analys64(pv, sd, nullptr, &vs, 2 * nb, OP_ANALYS, 0, s);
        if (e != cudaSuccess) break;
        k_vec64_join<<<dim3((unsigned)(pv.mmax + 1), (unsigned)nb), 128, 0, s>>>(pv, vs, (int)op);
        e = cudaGetLastError();
    }
    return e;
}

}  // namespace sht
