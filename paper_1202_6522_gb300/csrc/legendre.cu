// legendre.cu -- the FP32 Legendre stage of the Gauss-Legendre SHT on the CUDA
// cores, and the restart tables of both precisions (FP64: legendre64.cu).
//
// Synthesis (Sec. 2.2, Eq. synth_direct): for each order m and each latitude
// pair (x, -x), sum over n the spectral coefficients times P_n^m, split by the
// parity of n - m (mirror symmetry, Sec. 3.1):
//   E = sum_{n-m even} f_n^m P_n^m(x),  O = sum_{n-m odd} f_n^m P_n^m(x),
//   f_m(x) = E + O,  f_m(-x) = E - O   (the fold is applied by the FFT kernel).
// Analysis (Sec. 2.3, Eq. gauss): with s = w (F(x) + F(-x)), d = w (F(x) - F(-x))
// prepared by the FFT kernel, f_n^m = sum_pairs P_n^m(x) (s if n-m even else d).
//
// P_n^m is generated on the fly by the recurrence of Sec. 3.2, one latitude
// pair per lane, restarted at every segment of kSeedSeg degrees from the state
// the FP64 recurrence computed once per plan (the FP32 recurrence alone loses
// accuracy with n).  Underflow (Sec. 3.5) is taken care of per segment: where the
// values entering it are below 2^-63, the state is stored times a power of two
// that keeps the whole segment in the FP32 range, together with the factor that
// takes it back (0 where no |P| of the segment reaches 2^-70), so the recurrence
// itself tests nothing.  Since segments do not depend on one another, they are
// what the kernels split over warps.
//
// What bounds these kernels is instruction issue: 3 instructions of recurrence
// per degree and pair and 2 per field and degree, on the FMA pipe, plus
// whatever else the loops carry.  So a warp tests liveness and scaling once per
// segment, not per degree, and the sums over latitudes are taken across lanes
// once per segment of all pairs, not once per few degrees.
#include <cuda_runtime.h>

#include <climits>
#include <type_traits>

#include "sht_internal.h"

namespace sht {
namespace {

constexpr unsigned kFull = 0xffffffffu;

// P_n = a x P_{n-1} + b P_{n-2}.
__device__ __forceinline__ float next_p(float a, float b, float x, float y1, float y2)
{
    return fmaf(a * x, y1, b * y2);
}

// 16 bytes from global to shared memory, asynchronously; zeros unless `in`.
__device__ __forceinline__ void cp_async16(void *dst, const void *src, bool in)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(in ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N> __device__ __forceinline__ void cp_async_wait()
{
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// The kernels need the restart states and the tables of live groups.  A plan
// without them is refused rather than run on other arithmetic.
bool seeds_ok(const PlanView<float> &pv)
{
    return pv.segoff != nullptr && pv.seeds != nullptr && pv.glive != nullptr && pv.glive_vec != nullptr;
}

// Sums V values (a multiple of 32) over the 32 lanes and leaves lane l holding
// the sums of values [l V/32, (l + 1) V/32) in v[0 .. V/32).  Step by step a lane
// keeps half of its values and hands the other half to the lane O away.
template <int V, int O = 16, int N>
__device__ __forceinline__ void warp_transpose_reduce(float (&v)[N], int lane)
{
    if constexpr (O > 0) {
        constexpr int h = V / 2;
        const bool up = (lane & O) != 0;
#pragma unroll
        for (int q = 0; q < h; ++q) {
            const float send = up ? v[q] : v[q + h];
            const float keep = up ? v[q + h] : v[q];
            v[q] = keep + __shfl_xor_sync(kFull, send, O);
        }
        warp_transpose_reduce<h, O / 2>(v, lane);
    }
}

constexpr int kWarps = 4;   // warps per CTA of the kernels below

// Groups of 32 pairs of a plan.
__device__ __forceinline__ int groups_of(int npairs) { return (npairs + 31) >> 5; }

// ---------------------------------------------------------------------------
// Synthesis.  A CTA of four warps per (order m, block of 32 LPT pairs, BC
// fields): warp w sums the segments w, w + 4, ... over the block's pairs, LPT
// pairs per lane, and the warps' sums meet in shared memory in a fixed order.
// Which segments a warp takes does not depend on LPT, BC or the batch, nor does
// any sum.  Static polar optimisation (Sec. 3.1): a group of 32 pairs (one per
// lane) is left out of the segments before its first live one.
//
// Per degree, LPT pairs and BC fields: 3 LPT + 2 BC LPT FMA-pipe instructions,
// half a shared-memory load of (a, b) and BC / 2 of the spectral values, all
// broadcasts.  N = 2047, 2 fields: 552 us (issue 72 %, FMA pipe 45 %) against 817
// with a CTA of 256 pairs walking the degrees between barriers and testing each
// pair's scale at every degree; N = 383, 3-fold, 6 fields: 61 -> 13.5 us.
// ---------------------------------------------------------------------------
template <int LPT, int BC>
struct SynthSmem {
    float4 ab[kWarps][kSeedSeg / 2];          // (a, b) of two degrees
    float2 f[kWarps][kSeedSeg * BC];          // [degree][field]
    float4 sum[kWarps][LPT * 32 * BC];        // [pair][field] (E, O)
};

template <int LPT, int BC>
__device__ __forceinline__ void synth_tile(const PlanView<float> &pv, const float *__restrict__ spec,
                                           float *__restrict__ eo, int batch, int m, int pb, int b0, int op,
                                           SynthSmem<LPT, BC> &sm)
{
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int npairs = pv.npairs, ng = groups_of(npairs);
    const int L = pv.lmax - m * pv.mres + 1;   // order index m is the order m mres
    const int nseg = (L + kSeedSeg - 1) / kSeedSeg;
    const long col = col_of_mres(pv.lmax, m, pv.mres);
    const float2 *spec2 = reinterpret_cast<const float2 *>(spec);
    const float insc = (op == OP_ANALYS_ADJ && m > 0) ? 0.5f : 1.f;   // adjoint of analysis: b / c_m

    int p[LPT], gf[LPT], first = 0xffff;
    float x[LPT], er[LPT][BC], ei[LPT][BC], orr[LPT][BC], oi[LPT][BC];
#pragma unroll
    for (int i = 0; i < LPT; ++i) {
        const int g = pb * LPT + i;
        p[i] = g * 32 + lane;
        x[i] = p[i] < npairs ? pv.x[p[i]] : 0.f;
        gf[i] = g < ng ? (int)pv.glive[(size_t)m * ng + g] : 0xffff;
        first = min(first, gf[i]);
#pragma unroll
        for (int b = 0; b < BC; ++b) er[i][b] = ei[i][b] = orr[i][b] = oi[i][b] = 0.f;
    }

    // a segment's spectral values, (a, b) (lane = degree) and states (lane = pair),
    // read one segment ahead through pointers that step with the warp's segments
    int seg = first + ((w - first) & (kWarps - 1));   // the first one >= `first` of this warp
    if (seg > nseg) seg = nseg;
    const int nb = min(BC, batch - b0);
    const float2 *pab = pv.ab + col + seg * kSeedSeg + lane;
    const float2 *pf = spec2 + (size_t)b0 * pv.nlm + col + seg * kSeedSeg + lane;
    const float4 *ps = pv.seeds + (pv.segoff[m] + seg) * npairs + p[0];
    float2 nab, nf[BC];
    float4 ns[LPT];
    const auto fetch = [&](int sg) {
        const bool in = sg * kSeedSeg + lane < L;
        nab = in ? __ldg(pab) : make_float2(0.f, 0.f);
#pragma unroll
        for (int b = 0; b < BC; ++b) nf[b] = in && b < nb ? __ldg(pf + (size_t)b * pv.nlm) : make_float2(0.f, 0.f);
#pragma unroll
        for (int i = 0; i < LPT; ++i)
            ns[i] = sg < nseg && p[i] < npairs ? __ldg(ps + 32 * i) : make_float4(0.f, 0.f, 0.f, 0.f);
        pab += kWarps * kSeedSeg;
        pf += kWarps * kSeedSeg;
        ps += (size_t)kWarps * npairs;
    };
    fetch(seg);
    for (; seg < nseg; seg += kWarps) {
        const int cnt = min(kSeedSeg, L - seg * kSeedSeg);
        __syncwarp();   // the last segment's reads are done
        reinterpret_cast<float2 *>(sm.ab[w])[lane] = nab;
#pragma unroll
        for (int b = 0; b < BC; ++b)
            sm.f[w][lane * BC + b] = make_float2(nf[b].x * insc, m == 0 ? 0.f : nf[b].y * insc);
        float y1[LPT], y2[LPT], sc[LPT];
        bool all = true, scaled = false;
#pragma unroll
        for (int i = 0; i < LPT; ++i) {
            y1[i] = ns[i].x;
            y2[i] = ns[i].y;
            sc[i] = ns[i].z;
            all = all && seg >= gf[i];
            scaled = scaled || (sc[i] != 1.f && p[i] < npairs);
        }
        fetch(seg + kWarps);
        __syncwarp();
        if (all && !__any_sync(kFull, scaled)) {
#pragma unroll 1
            for (int tb = 0; tb < cnt; tb += 8)   // rows past cnt are zero
#pragma unroll
            for (int t = tb; t < tb + 8; t += 2) {
                const float4 ab = sm.ab[w][t >> 1];
#pragma unroll
                for (int i = 0; i < LPT; ++i) y2[i] = next_p(ab.x, ab.y, x[i], y1[i], y2[i]);
#pragma unroll
                for (int b = 0; b < BC; ++b) {
                    const float2 f = sm.f[w][t * BC + b];
#pragma unroll
                    for (int i = 0; i < LPT; ++i) {
                        er[i][b] = fmaf(f.x, y2[i], er[i][b]);
                        ei[i][b] = fmaf(f.y, y2[i], ei[i][b]);
                    }
                }
#pragma unroll
                for (int i = 0; i < LPT; ++i) y1[i] = next_p(ab.z, ab.w, x[i], y2[i], y1[i]);
#pragma unroll
                for (int b = 0; b < BC; ++b) {
                    const float2 f = sm.f[w][(t + 1) * BC + b];
#pragma unroll
                    for (int i = 0; i < LPT; ++i) {
                        orr[i][b] = fmaf(f.x, y1[i], orr[i][b]);
                        oi[i][b] = fmaf(f.y, y1[i], oi[i][b]);
                    }
                }
            }
        } else {
            // a group not live yet, or a pair whose state is stored scaled
#pragma unroll
            for (int i = 0; i < LPT; ++i) {
                if (seg < gf[i]) continue;
#pragma unroll 2
                for (int t = 0; t < cnt; t += 2) {
                    const float4 ab = sm.ab[w][t >> 1];
                    y2[i] = next_p(ab.x, ab.y, x[i], y1[i], y2[i]);
                    const float c0 = sc[i] * y2[i];
                    y1[i] = next_p(ab.z, ab.w, x[i], y2[i], y1[i]);
                    const float c1 = sc[i] * y1[i];
#pragma unroll
                    for (int b = 0; b < BC; ++b) {
                        const float2 f0 = sm.f[w][t * BC + b], f1 = sm.f[w][(t + 1) * BC + b];
                        er[i][b] = fmaf(f0.x, c0, er[i][b]);
                        ei[i][b] = fmaf(f0.y, c0, ei[i][b]);
                        orr[i][b] = fmaf(f1.x, c1, orr[i][b]);
                        oi[i][b] = fmaf(f1.y, c1, oi[i][b]);
                    }
                }
            }
        }
    }
#pragma unroll
    for (int i = 0; i < LPT; ++i)
#pragma unroll
        for (int b = 0; b < BC; ++b)
            sm.sum[w][(b * LPT + i) * 32 + lane] = make_float4(er[i][b], ei[i][b], orr[i][b], oi[i][b]);
    __syncthreads();
    float4 *eo4 = reinterpret_cast<float4 *>(eo);
    for (int q = threadIdx.x; q < LPT * 32 * BC; q += 32 * kWarps) {
        const int b = q / (LPT * 32), pp = pb * LPT * 32 + q % (LPT * 32);
        if (b0 + b >= batch || pp >= npairs) continue;
        float4 v = sm.sum[0][q];
#pragma unroll
        for (int u = 1; u < kWarps; ++u) {
            const float4 z = sm.sum[u][q];
            v.x += z.x; v.y += z.y; v.z += z.z; v.w += z.w;
        }
        eo4[((size_t)(b0 + b) * (pv.mmax + 1) + m) * npairs + pp] = v;
    }
}

// blockIdx.x = (m, pair block), heaviest m first; blockIdx.y = field chunk.
template <int LPT, int BC>
__global__ void __launch_bounds__(32 * kWarps)
k_synth(PlanView<float> pv, const float *__restrict__ spec, float *__restrict__ eo, int batch, int npb, int op)
{
    __shared__ SynthSmem<LPT, BC> sm;
    const int m = blockIdx.x / npb, pb = blockIdx.x - m * npb;
    synth_tile<LPT, BC>(pv, spec, eo, batch, m, pb, blockIdx.y * BC, op, sm);
}

// First group of 32 pairs with a live pair in segment `seg` (the group count if
// there is none), warp-uniform.  glive: first live segment of each group.
__device__ __forceinline__ int first_live_group(const unsigned short *__restrict__ glive, int ng, int seg, int lane)
{
    for (int gb = 0; gb < ng; gb += 32) {
        const bool lv = gb + lane < ng && (int)glive[gb + lane] <= seg;
        const unsigned mk = __ballot_sync(kFull, lv);
        if (mk) return gb + __ffs(mk) - 1;
    }
    return ng;
}

// ---------------------------------------------------------------------------
// Analysis of one segment of order m by one warp, over all latitude pairs, BC
// fields.  A lane takes the pairs lane, lane + 32, ... one after the other: it
// restarts the recurrence and adds P_n (s or d) into one accumulator per
// degree, field and part, 64 BC of them; one butterfly at the end sums them
// over the lanes and leaves lane t the sums of degree t.  Per degree and pair 3
// instructions of recurrence, 2 BC of sums and half a load of (a, b); the
// butterfly (~4 instructions per accumulator) is shared by all pairs.  States and
// folds come kRing pairs ahead by asynchronous copies into slots of the lane's
// own (the accumulators leave 12 warps per SM, too few to cover a DRAM access
// with one pair's sums).  Pairs come in a fixed order, so results are bitwise
// reproducible.  N = 2047, 2 fields: 560 us (issue 67 %) against 2106 with a CTA
// per order that reduced over its lanes and warps every 8 degrees; the same form
// with plain loads one pair ahead took 1536.  N = 383, 3-fold, 6 fields: 89 -> 14 us.
// ---------------------------------------------------------------------------
constexpr int kRing = 4;

template <int BC>
struct AnalysSmem {
    float4 ab[kSeedSeg / 2];          // (a, b) of two degrees
    float4 ring[kRing][1 + BC][32];   // state; folds (s, d) of each field
};

template <int BC>
__device__ __forceinline__ void analys_segment(const PlanView<float> &pv, const float *__restrict__ sd,
                                               float *__restrict__ spec, int batch, int m, int seg, int b0, int op,
                                               AnalysSmem<BC> &sm)
{
    constexpr int C = 2 * BC;
    const int lane = threadIdx.x & 31;
    const int npairs = pv.npairs, ng = groups_of(npairs);
    const int L = pv.lmax - m * pv.mres + 1;
    const int n0 = seg * kSeedSeg, cnt = min(kSeedSeg, L - n0);
    const long col = col_of_mres(pv.lmax, m, pv.mres) + n0;
    const float4 *sd4 = reinterpret_cast<const float4 *>(sd) + ((size_t)b0 * (pv.mmax + 1) + m) * npairs;
    const size_t fstride = (size_t)(pv.mmax + 1) * npairs;

    const int g0 = first_live_group(pv.glive + (size_t)m * ng, ng, seg, lane);
    // the next pair to fetch (pointers stop at the lane's last pair) and its slot
    int p = g0 * 32 + lane, slot = 0;
    const int q0 = min(p, npairs - 1), nb = min(BC, batch - b0);
    const float4 *ps = pv.seeds + (pv.segoff[m] + seg) * npairs + q0, *pf = sd4 + q0;
    const float *px = pv.x + q0;
    const auto fetch = [&]() {   // one group of copies per call, also past the last pair
        const bool in = p < npairs;
        cp_async16(&sm.ring[slot][0][lane], ps, in);
#pragma unroll
        for (int b = 0; b < BC; ++b) cp_async16(&sm.ring[slot][1 + b][lane], pf + (b < nb ? b * fstride : 0), in && b < nb);
        cp_async_commit();
        p += 32;
        slot = (slot + 1) & (kRing - 1);
        const int step = p < npairs ? 32 : 0;
        ps += step;
        pf += step;
    };
#pragma unroll
    for (int u = 0; u < kRing - 1; ++u) fetch();
    __syncwarp();   // the last segment is done with sm.ab
    reinterpret_cast<float2 *>(sm.ab)[lane] = lane < cnt ? __ldg(pv.ab + col + lane) : make_float2(0.f, 0.f);
    __syncwarp();

    float acc[kSeedSeg * C];
#pragma unroll
    for (int q = 0; q < kSeedSeg * C; ++q) acc[q] = 0.f;
#pragma unroll 1
    for (int g = g0; g < ng; ++g) {
        const float x = __ldg(px);
        px += (g + 1) * 32 + lane < npairs ? 32 : 0;
        cp_async_wait<kRing - 2>();
        const float4 (&r)[1 + BC][32] = sm.ring[(slot + 1) & (kRing - 1)];   // the oldest
        const float4 st = r[0][lane];
        float4 f[BC];
#pragma unroll
        for (int b = 0; b < BC; ++b) f[b] = r[1 + b][lane];
        fetch();
        float y1 = st.x, y2 = st.y;
        // one group of pairs; `scaled`: P = factor y
        const auto add = [&](auto scaled) {
            constexpr bool kScaled = decltype(scaled)::value;
#pragma unroll
            for (int tb = 0; tb < kSeedSeg; tb += 8) {
                if (tb >= cnt) break;   // rows past cnt are zero
#pragma unroll
                for (int t = tb; t < tb + 8; t += 2) {
                    const float4 ab = sm.ab[t >> 1];
                    y2 = next_p(ab.x, ab.y, x, y1, y2);
                    y1 = next_p(ab.z, ab.w, x, y2, y1);
                    const float c0 = kScaled ? y2 * st.z : y2, c1 = kScaled ? y1 * st.z : y1;
#pragma unroll
                    for (int b = 0; b < BC; ++b) {
                        float *a = acc + t * C + 2 * b;
                        a[0] = fmaf(c0, f[b].x, a[0]);
                        a[1] = fmaf(c0, f[b].y, a[1]);
                        a[C] = fmaf(c1, f[b].z, a[C]);
                        a[C + 1] = fmaf(c1, f[b].w, a[C + 1]);
                    }
                }
            }
        };
        // the factor goes to P, not to the folds: times the folds of small data it leaves
        // the FP32 range, though P times fold does not
        if (__any_sync(kFull, st.z != 1.f)) add(std::true_type());
        else add(std::false_type());
    }
    cp_async_wait<0>();
    warp_transpose_reduce<kSeedSeg * C>(acc, lane);
    if (lane >= cnt) return;
    const float outsc = (op == OP_SYNTH_ADJ && m > 0) ? 2.f : 1.f;   // c_m for the adjoint of synthesis
    float2 *spec2 = reinterpret_cast<float2 *>(spec);
#pragma unroll
    for (int b = 0; b < BC; ++b) {
        if (b0 + b >= batch) break;
        spec2[(size_t)(b0 + b) * pv.nlm + col + lane] =
            make_float2(acc[2 * b] * outsc, m == 0 ? 0.f : acc[2 * b + 1] * outsc);
    }
}

// blockIdx: x four segments (a warp each; neighbours of one order share its
// folds in L1), y order index, z field chunk.
template <int BC>
__global__ void __launch_bounds__(32 * kWarps)
k_analys(PlanView<float> pv, const float *__restrict__ sd, float *__restrict__ spec, int batch, int op)
{
    __shared__ AnalysSmem<BC> sm[kWarps];
    const int w = threadIdx.x >> 5, seg = blockIdx.x * kWarps + w, m = blockIdx.y;
    if (seg * kSeedSeg > pv.lmax - m * pv.mres) return;
    analys_segment<BC>(pv, sd, spec, batch, m, seg, blockIdx.z * BC, op, sm[w]);
}

// ---------------------------------------------------------------------------
// Vector synthesis.  With dP = sin(theta) dP/dtheta = n x P_n - dc_n P_{n-1}:
//   sin * V_theta,m = sum [S dP - i m T P],   sin * V_phi,m = sum [i m S P + T dP].
// dP has the opposite mirror parity of P, so a degree with n - m even adds its
// P terms to E and its dP terms to O, an odd one the other way round: four
// complex sums per pair and field (theta and phi, E and O), the factors -i m and
// i m taken into the spectral values.  CTA and warps as in the scalar synthesis;
// a group of 32 pairs is left out of the segments in which none of its values
// reaches 2^-70.  Per degree and pair 6 instructions for P and dP and 8 per
// field; N = 511, 8 fields: 193 -> 144 us (issue 63 %, FMA pipe 46 %).
// ---------------------------------------------------------------------------
template <int LPT, int BC>
struct SynthVecSmem {
    float4 rec[kWarps][kSeedSeg];                   // (a, b, dc, n)
    float4 f[kWarps][kSeedSeg * BC][2];             // [degree][field] (S, T), (-i m T, i m S)
    float4 sum[kWarps][LPT * 32 * BC];              // [pair][field] (E, O) of one component
};

// P and dP of the degree of r.
__device__ __forceinline__ void vec_step(const float4 &r, float x, float &y1, float &y2, float &c, float &cd)
{
    c = next_p(r.x, r.y, x, y1, y2);
    y2 = y1;
    y1 = c;
    cd = fmaf(r.w * x, y1, -r.z * y2);
}

// Adds one degree of one field to a pair's sums: P terms to the component of
// the degree's parity, dP terms to the other.
template <bool ODD>
__device__ __forceinline__ void vec_add(const float4 (&f)[2], float c, float cd, float (&te)[2], float (&to)[2],
                                        float (&pe)[2], float (&po)[2])
{
    float (&tp)[2] = ODD ? to : te, (&td)[2] = ODD ? te : to;
    float (&pp)[2] = ODD ? po : pe, (&pd)[2] = ODD ? pe : po;
    tp[0] = fmaf(f[1].x, c, tp[0]);
    tp[1] = fmaf(f[1].y, c, tp[1]);
    pp[0] = fmaf(f[1].z, c, pp[0]);
    pp[1] = fmaf(f[1].w, c, pp[1]);
    td[0] = fmaf(f[0].x, cd, td[0]);
    td[1] = fmaf(f[0].y, cd, td[1]);
    pd[0] = fmaf(f[0].z, cd, pd[0]);
    pd[1] = fmaf(f[0].w, cd, pd[1]);
}

template <int LPT, int BC>
__global__ void __launch_bounds__(32 * kWarps)
k_synth_vec(PlanView<float> pv, const float *__restrict__ Sg, const float *__restrict__ Tg, float *__restrict__ eot,
            float *__restrict__ eop, int batch, int npb, int op)
{
    __shared__ SynthVecSmem<LPT, BC> sm;
    const int m = blockIdx.x / npb, pb = blockIdx.x - m * npb, b0 = blockIdx.y * BC;
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int npairs = pv.npairs, ng = groups_of(npairs);
    const int L = pv.lmax - m * pv.mres + 1;
    const int nseg = (L + kSeedSeg - 1) / kSeedSeg;
    const long col = col_of_mres(pv.lmax, m, pv.mres);
    const float2 *S2 = reinterpret_cast<const float2 *>(Sg), *T2 = reinterpret_cast<const float2 *>(Tg);
    const float cadj = (op == OP_ANALYS_ADJ && m > 0) ? 0.5f : 1.f, fm = (float)(m * pv.mres);

    int p[LPT], gf[LPT], first = 0xffff;
    float x[LPT], te[LPT][BC][2], to[LPT][BC][2], pe[LPT][BC][2], po[LPT][BC][2];   // theta and phi, E and O
#pragma unroll
    for (int i = 0; i < LPT; ++i) {
        const int g = pb * LPT + i;
        p[i] = g * 32 + lane;
        x[i] = p[i] < npairs ? pv.x[p[i]] : 0.f;
        gf[i] = g < ng ? (int)pv.glive_vec[(size_t)m * ng + g] : 0xffff;
        first = min(first, gf[i]);
#pragma unroll
        for (int b = 0; b < BC; ++b)
#pragma unroll
            for (int q = 0; q < 2; ++q) te[i][b][q] = to[i][b][q] = pe[i][b][q] = po[i][b][q] = 0.f;
    }
    for (int seg = first + ((w - first) & (kWarps - 1)); seg < nseg; seg += kWarps) {
        const int cnt = min(kSeedSeg, L - seg * kSeedSeg), t0 = seg * kSeedSeg + lane, n = m * pv.mres + t0;
        float y1[LPT], y2[LPT], fac[LPT];
        bool all = true, scaled = false;
#pragma unroll
        for (int i = 0; i < LPT; ++i) {
            const float4 s = p[i] < npairs ? __ldg(pv.seeds + (pv.segoff[m] + seg) * npairs + p[i])
                                           : make_float4(0.f, 0.f, 0.f, 0.f);
            y1[i] = s.x;
            y2[i] = s.y;
            fac[i] = s.z;
            all = all && seg >= gf[i];
            scaled = scaled || (fac[i] != 1.f && p[i] < npairs);
        }
        __syncwarp();
        float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
        if (lane < cnt) {
            const float2 ab = __ldg(pv.ab + col + t0);
            r = make_float4(ab.x, ab.y, __ldg(pv.dc + col + t0), (float)n);
        }
        sm.rec[w][lane] = r;
        // adjoint of analysis: b / (c_m n(n+1)), nothing at n = 0
        float sc = 1.f;
        if (op == OP_ANALYS_ADJ) sc = (n == 0) ? 0.f : cadj / ((float)n * (float)(n + 1));
#pragma unroll
        for (int b = 0; b < BC; ++b) {
            float2 s = make_float2(0.f, 0.f), t = s;
            if (lane < cnt && b0 + b < batch) {
                s = __ldg(S2 + (size_t)(b0 + b) * pv.nlm + col + t0);
                t = __ldg(T2 + (size_t)(b0 + b) * pv.nlm + col + t0);
                s = make_float2(s.x * sc, m == 0 ? 0.f : s.y * sc);
                t = make_float2(t.x * sc, m == 0 ? 0.f : t.y * sc);
            }
            sm.f[w][lane * BC + b][0] = make_float4(s.x, s.y, t.x, t.y);
            sm.f[w][lane * BC + b][1] = make_float4(fm * t.y, -fm * t.x, -fm * s.y, fm * s.x);
        }
        __syncwarp();
        if (all && !__any_sync(kFull, scaled)) {
#pragma unroll 1
            for (int tb = 0; tb < cnt; tb += 4)   // rows past cnt are zero
#pragma unroll
            for (int t = tb; t < tb + 4; t += 2) {
                float c[LPT], cd[LPT];
#pragma unroll
                for (int i = 0; i < LPT; ++i) vec_step(sm.rec[w][t], x[i], y1[i], y2[i], c[i], cd[i]);
#pragma unroll
                for (int b = 0; b < BC; ++b)
#pragma unroll
                    for (int i = 0; i < LPT; ++i)
                        vec_add<false>(sm.f[w][t * BC + b], c[i], cd[i], te[i][b], to[i][b], pe[i][b], po[i][b]);
#pragma unroll
                for (int i = 0; i < LPT; ++i) vec_step(sm.rec[w][t + 1], x[i], y1[i], y2[i], c[i], cd[i]);
#pragma unroll
                for (int b = 0; b < BC; ++b)
#pragma unroll
                    for (int i = 0; i < LPT; ++i)
                        vec_add<true>(sm.f[w][(t + 1) * BC + b], c[i], cd[i], te[i][b], to[i][b], pe[i][b], po[i][b]);
            }
        } else {
            // a group not live yet, or a pair whose state is stored scaled
#pragma unroll
            for (int i = 0; i < LPT; ++i) {
                if (seg < gf[i]) continue;
                for (int t = 0; t < cnt; t += 2) {
                    float c, cd;
                    vec_step(sm.rec[w][t], x[i], y1[i], y2[i], c, cd);
                    c *= fac[i];
                    cd *= fac[i];
#pragma unroll
                    for (int b = 0; b < BC; ++b)
                        vec_add<false>(sm.f[w][t * BC + b], c, cd, te[i][b], to[i][b], pe[i][b], po[i][b]);
                    vec_step(sm.rec[w][t + 1], x[i], y1[i], y2[i], c, cd);
                    c *= fac[i];
                    cd *= fac[i];
#pragma unroll
                    for (int b = 0; b < BC; ++b)
                        vec_add<true>(sm.f[w][(t + 1) * BC + b], c, cd, te[i][b], to[i][b], pe[i][b], po[i][b]);
                }
            }
        }
    }
    // the warps' sums, theta then phi, divided by sin(theta)
#pragma unroll
    for (int comp = 0; comp < 2; ++comp) {
        __syncthreads();
#pragma unroll
        for (int i = 0; i < LPT; ++i)
#pragma unroll
            for (int b = 0; b < BC; ++b)
                sm.sum[w][(b * LPT + i) * 32 + lane] =
                    comp == 0 ? make_float4(te[i][b][0], te[i][b][1], to[i][b][0], to[i][b][1])
                              : make_float4(pe[i][b][0], pe[i][b][1], po[i][b][0], po[i][b][1]);
        __syncthreads();
        float4 *eo4 = reinterpret_cast<float4 *>(comp == 0 ? eot : eop);
        for (int q = threadIdx.x; q < LPT * 32 * BC; q += 32 * kWarps) {
            const int b = q / (LPT * 32), pp = pb * LPT * 32 + q % (LPT * 32);
            if (b0 + b >= batch || pp >= npairs) continue;
            const float is = 1.f / pv.st[pp];
            float4 v = sm.sum[0][q];
#pragma unroll
            for (int u = 1; u < kWarps; ++u) {
                const float4 z = sm.sum[u][q];
                v.x += z.x; v.y += z.y; v.z += z.z; v.w += z.w;
            }
            eo4[((size_t)(b0 + b) * (pv.mmax + 1) + m) * npairs + pp] =
                make_float4(v.x * is, v.y * is, v.z * is, v.w * is);
        }
    }
}

// ---------------------------------------------------------------------------
// Vector analysis.  With folds s/d of (w/sin) V_theta and V_phi:
//   S_n = sum [dP * fold(V_theta) - i m P * fold(V_phi)] / (n(n+1))
//   T_n = sum [i m P * fold(V_theta) + dP * fold(V_phi)] / (n(n+1))
// where the fold is s for an even function and d for an odd one.  A warp per
// segment and field, as in the scalar analysis: four accumulators per degree
// (S and T), the folds times m beside the folds.  N = 511, 8 fields: 452 -> 215 us.
// ---------------------------------------------------------------------------
struct AnalysVecSmem {
    float4 rec[kSeedSeg];         // (a, b, dc, n)
    float4 ring[kRing][3][32];    // state; folds (s, d) of theta and phi
};

__global__ void __launch_bounds__(32 * kWarps)
k_analys_vec(PlanView<float> pv, const float *__restrict__ sdt, const float *__restrict__ sdp, float *__restrict__ So,
             float *__restrict__ To, int op)
{
    __shared__ AnalysVecSmem s_sm[kWarps];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int seg = blockIdx.x * kWarps + w, m = blockIdx.y, b = blockIdx.z;
    const int npairs = pv.npairs, ng = groups_of(npairs);
    const int L = pv.lmax - m * pv.mres + 1;
    const int n0 = seg * kSeedSeg;
    if (n0 >= L) return;
    AnalysVecSmem &sm = s_sm[w];
    const int cnt = min(kSeedSeg, L - n0), n = m * pv.mres + n0 + lane;
    const long col = col_of_mres(pv.lmax, m, pv.mres) + n0;
    const float fm = (float)(m * pv.mres);
    const int g0 = first_live_group(pv.glive_vec + (size_t)m * ng, ng, seg, lane);
    int p = g0 * 32 + lane, slot = 0;   // as in analys_segment
    const int q0 = min(p, npairs - 1);
    const float4 *ps = pv.seeds + (pv.segoff[m] + seg) * npairs + q0;
    const size_t fo = ((size_t)b * (pv.mmax + 1) + m) * npairs + q0;
    const float4 *ft = reinterpret_cast<const float4 *>(sdt) + fo, *fp = reinterpret_cast<const float4 *>(sdp) + fo;
    const float *px = pv.x + q0;
    const auto fetch = [&]() {
        const bool in = p < npairs;
        cp_async16(&sm.ring[slot][0][lane], ps, in);
        cp_async16(&sm.ring[slot][1][lane], ft, in);
        cp_async16(&sm.ring[slot][2][lane], fp, in);
        cp_async_commit();
        p += 32;
        slot = (slot + 1) & (kRing - 1);
        const int step = p < npairs ? 32 : 0;
        ps += step;
        ft += step;
        fp += step;
    };
#pragma unroll
    for (int u = 0; u < kRing - 1; ++u) fetch();
    {
        float4 r = make_float4(0.f, 0.f, 0.f, 0.f);
        if (lane < cnt) {
            const float2 ab = __ldg(pv.ab + col + lane);
            r = make_float4(ab.x, ab.y, __ldg(pv.dc + col + lane), (float)n);
        }
        sm.rec[lane] = r;
    }
    __syncwarp();

    float acc[kSeedSeg * 4];   // per degree: S, T
#pragma unroll
    for (int q = 0; q < kSeedSeg * 4; ++q) acc[q] = 0.f;
#pragma unroll 1
    for (int g = g0; g < ng; ++g) {
        const float x = __ldg(px);
        px += (g + 1) * 32 + lane < npairs ? 32 : 0;
        cp_async_wait<kRing - 2>();
        const float4 (&r)[3][32] = sm.ring[(slot + 1) & (kRing - 1)];   // the oldest
        const float4 st = r[0][lane];
        const float4 vt = r[1][lane], vp = r[2][lane];   // (s, d) of theta and phi
        fetch();
        float y1 = st.x, y2 = st.y;
        const float4 mt = make_float4(fm * vt.x, fm * vt.y, fm * vt.z, fm * vt.w);
        const float4 mp = make_float4(fm * vp.x, fm * vp.y, fm * vp.z, fm * vp.w);
        const auto add = [&](auto scaled) {   // as in analys_segment
            constexpr bool kScaled = decltype(scaled)::value;
#pragma unroll
            for (int tb = 0; tb < kSeedSeg; tb += 8) {
                if (tb >= cnt) break;   // rows past cnt are zero
#pragma unroll
                for (int t = tb; t < tb + 8; ++t) {
                    float c, cd;
                    vec_step(sm.rec[t], x, y1, y2, c, cd);
                    if (kScaled) {
                        c *= st.z;
                        cd *= st.z;
                    }
                    // n - m even: P even -> s folds, dP odd -> d folds; odd: the other way round
                    const bool odd = t & 1;
                    float *a = acc + 4 * t;
                    a[0] = fmaf(cd, odd ? vt.x : vt.z, fmaf(c, odd ? mp.w : mp.y, a[0]));
                    a[1] = fmaf(cd, odd ? vt.y : vt.w, fmaf(-c, odd ? mp.z : mp.x, a[1]));
                    a[2] = fmaf(cd, odd ? vp.x : vp.z, fmaf(-c, odd ? mt.w : mt.y, a[2]));
                    a[3] = fmaf(cd, odd ? vp.y : vp.w, fmaf(c, odd ? mt.z : mt.x, a[3]));
                }
            }
        };
        if (__any_sync(kFull, st.z != 1.f)) add(std::true_type());   // states stored scaled: P = factor y
        else add(std::false_type());
    }
    cp_async_wait<0>();
    warp_transpose_reduce<kSeedSeg * 4>(acc, lane);
    if (lane >= cnt) return;
    float sc;
    if (op == OP_SYNTH_ADJ) sc = (m > 0) ? 2.f : 1.f;
    else sc = (n == 0) ? 0.f : 1.f / ((float)n * (float)(n + 1));
    const size_t o = (size_t)b * pv.nlm + col + lane;
    reinterpret_cast<float2 *>(So)[o] = make_float2(sc * acc[0], m == 0 ? 0.f : sc * acc[1]);
    reinterpret_cast<float2 *>(To)[o] = make_float2(sc * acc[2], m == 0 ? 0.f : sc * acc[3]);
}

// Field chunk per CTA for a batch.
inline int pick_bc(int batch) { return batch >= 4 ? 4 : (batch >= 2 ? 2 : 1); }

inline unsigned segment_ctas(const PlanView<float> &pv)
{
    return (unsigned)((pv.lmax + kSeedSeg * kWarps) / (kSeedSeg * kWarps));
}

template <int LPT, int BC>
cudaError_t synth_go(const PlanView<float> &pv, const float *spec, float *eo, int batch, Op op, cudaStream_t s)
{
    const int npb = (pv.npairs + 32 * LPT - 1) / (32 * LPT);
    dim3 grid((unsigned)((pv.mmax + 1) * npb), (unsigned)((batch + BC - 1) / BC));
    k_synth<LPT, BC><<<grid, 32 * kWarps, 0, s>>>(pv, spec, eo, batch, npb, (int)op);
    return cudaGetLastError();
}

template <int BC>
cudaError_t analys_go(const PlanView<float> &pv, const float *sd, float *spec, int batch, Op op, cudaStream_t s)
{
    dim3 grid(segment_ctas(pv), (unsigned)(pv.mmax + 1), (unsigned)((batch + BC - 1) / BC));
    k_analys<BC><<<grid, 32 * kWarps, 0, s>>>(pv, sd, spec, batch, (int)op);
    return cudaGetLastError();
}

template <int LPT, int BC>
cudaError_t synth_vec_go(const PlanView<float> &pv, const float *S, const float *Tc, float *eot, float *eop, int batch,
                         Op op, cudaStream_t s)
{
    const int npb = (pv.npairs + 32 * LPT - 1) / (32 * LPT);
    dim3 grid((unsigned)((pv.mmax + 1) * npb), (unsigned)((batch + BC - 1) / BC));
    k_synth_vec<LPT, BC><<<grid, 32 * kWarps, 0, s>>>(pv, S, Tc, eot, eop, batch, npb, (int)op);
    return cudaGetLastError();
}

}  // namespace

cudaError_t launch_legendre_synth(const PlanView<float> &pv, const float *spec, float *eo, int batch, Op op, int lpt,
                                  int bc, cudaStream_t s)
{
    if (!seeds_ok(pv)) return cudaErrorInvalidValue;
    // default shape: 2 pairs per lane, up to 4 fields per CTA
    if (lpt <= 0) lpt = 2;
    if (bc <= 0) bc = pick_bc(batch);
#define SHT_SYN(L, B) if (lpt == L && bc == B) return synth_go<L, B>(pv, spec, eo, batch, op, s);
    SHT_SYN(1, 1) SHT_SYN(1, 2) SHT_SYN(1, 4)
    SHT_SYN(2, 1) SHT_SYN(2, 2) SHT_SYN(2, 4)
    SHT_SYN(4, 1) SHT_SYN(4, 2)
#undef SHT_SYN
    return cudaErrorInvalidValue;
}

cudaError_t launch_legendre_analys(const PlanView<float> &pv, const float *sd, float *spec, int batch, Op op, int bc,
                                   cudaStream_t s)
{
    if (!seeds_ok(pv)) return cudaErrorInvalidValue;
    if (bc <= 0) bc = batch >= 2 ? 2 : 1;
    if (bc == 1) return analys_go<1>(pv, sd, spec, batch, op, s);
    if (bc == 2) return analys_go<2>(pv, sd, spec, batch, op, s);
    return cudaErrorInvalidValue;
}

cudaError_t launch_legendre_synth_vec(const PlanView<float> &pv, const float *S, const float *Tc, float *eot,
                                      float *eop, int batch, Op op, cudaStream_t s)
{
    if (!seeds_ok(pv)) return cudaErrorInvalidValue;
    if (batch >= 2) return synth_vec_go<2, 2>(pv, S, Tc, eot, eop, batch, op, s);
    return synth_vec_go<2, 1>(pv, S, Tc, eot, eop, batch, op, s);
}

cudaError_t launch_legendre_analys_vec(const PlanView<float> &pv, const float *sdt, const float *sdp, float *S,
                                       float *Tc, int batch, Op op, cudaStream_t s)
{
    if (!seeds_ok(pv)) return cudaErrorInvalidValue;
    dim3 grid(segment_ctas(pv), (unsigned)(pv.mmax + 1), (unsigned)batch);
    k_analys_vec<<<grid, 32 * kWarps, 0, s>>>(pv, sdt, sdp, S, Tc, (int)op);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Persistent kernels for uneven batches (one field per tile).
// ---------------------------------------------------------------------------
namespace {

__global__ void __launch_bounds__(32 * kWarps) k_batch_synth(const BatchField *__restrict__ fields,
                                                             const int4 *__restrict__ tiles, int ntiles, int *counter)
{
    __shared__ SynthSmem<2, 1> sm;
    __shared__ int s_tile;
    for (;;) {
        __syncthreads();  // the previous tile is done with the shared buffers
        if (threadIdx.x == 0) s_tile = atomicAdd(counter, 1);
        __syncthreads();
        const int t = s_tile;
        if (t >= ntiles) break;
        const int4 tl = tiles[t];
        const BatchField f = fields[tl.x];
        synth_tile<2, 1>(f.pv, f.in, f.inter, 1, tl.y, tl.z, 0, OP_SYNTH, sm);
    }
}

// A warp takes the next four segments of an order at a time.
__global__ void __launch_bounds__(32 * kWarps) k_batch_analys(const BatchField *__restrict__ fields,
                                                              const int4 *__restrict__ tiles, int ntiles, int *counter)
{
    __shared__ AnalysSmem<1> sm[kWarps];
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (;;) {
        int t = 0;
        if (lane == 0) t = atomicAdd(counter, 1);
        t = __shfl_sync(kFull, t, 0);
        if (t >= ntiles) break;
        const int4 tl = tiles[t];
        const BatchField f = fields[tl.x];
        const int nseg = (f.pv.lmax - tl.y * f.pv.mres + kSeedSeg) / kSeedSeg;
        for (int seg = tl.z; seg < min(nseg, tl.z + kBatchAnalysSegs); ++seg)
            analys_segment<1>(f.pv, f.inter, f.out, 1, tl.y, seg, 0, OP_ANALYS, sm[w]);
    }
}

}  // namespace

cudaError_t launch_batch_legendre(bool synth, const BatchField *fields, const int4 *tiles, int ntiles, int *counter,
                                  int ctas, cudaStream_t s)
{
    if (synth) k_batch_synth<<<ctas, 32 * kWarps, 0, s>>>(fields, tiles, ntiles, counter);
    else k_batch_analys<<<ctas, 32 * kWarps, 0, s>>>(fields, tiles, ntiles, counter);
    return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Restart states of the recurrence and the first-live table of the static
// polar optimisation.  One thread per (order index m, pair): the FP64
// recurrence of Sec. 3.2 from P_m^m, carried as y 2^(-240 k) (Sec. 3.5).  At
// the start of every kSeedSeg-degree segment the state (y1, y2) =
// (P_{n0-1}, P_{n0-2}) is stored: times 2^hseg with k (FP64 plans), or in the
// form of the FP32 kernels, (y1, y2, factor) with P = factor y (fp32_state).
// live[m][pair] is the first segment that holds a degree with |P_n^m| >= thr to
// within 2^-20 of its value (all segments live when thr <= 0; the segment count
// when none is), glive the smallest of each group of 32 pairs, and glive_vec the
// group's first segment that holds a value the precision keeps (2^-70 in FP32; any
// unscaled one in FP64): segments that contribute nothing at any threshold.
// The kernel is bound by its FP64 instructions, three per degree: every test is
// on the high words (22 -> 13 ms at N = 2047 with FP64 comparisons left out).
// ---------------------------------------------------------------------------
namespace {

constexpr int kLeast32 = -70;   // FP32 leaves out segments with every |P| below 2^kLeast32

// y 2^(-240 k) = P; emax: floor(log2) of the segment's largest |P|.  A state of
// at least 2^-63 is stored as it is.  A smaller one can grow by up to 2^149 over
// 32 degrees (order 4095): it is stored times the power of two that takes the
// segment's largest value to about 2^50, which leaves every value and the factor
// in FP32's normal range; the recurrence rounds the same at either scale.
// Exponents from the high words and powers of two from integers: the FP64 pipe is
// left to the recurrence.
__device__ float4 fp32_state(double y1, double y2, int k, int emax)
{
    constexpr int kTop = 50;
    const int h = max(__double2hiint(y1) & 0x7fffffff, __double2hiint(y2) & 0x7fffffff);
    if (h < 0x100000 || emax < kLeast32) return make_float4(0.f, 0.f, 0.f, 0.f);
    const int down = -Scale<double>::S * k;
    if (k == 0 && (h >> 20) - 1023 >= -63) return make_float4((float)y1, (float)y2, 1.f, 0.f);
    // 0 below FP64's range, where the states are below FP32's all the same
    const int e = kTop - emax, field = 1023 + down + e;
    const double f = field > 0 ? __hiloint2double(min(field, 2046) << 20, 0) : 0.0;
    return make_float4((float)(y1 * f), (float)(y2 * f), __int_as_float((127 - e) << 23), 0.f);
}

__global__ void __launch_bounds__(128)
k_build_restarts(PlanView<double> pv, const unsigned long long *__restrict__ segoff, float4 *__restrict__ seeds32,
                 double2 *__restrict__ seeds64, int *__restrict__ seeds64k, const int *__restrict__ hseg,
                 unsigned short *__restrict__ live, unsigned short *__restrict__ glive,
                 unsigned short *__restrict__ glive_vec, double thr)
{
    const int m = blockIdx.y;
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    const int npairs = pv.npairs;
    const bool in = p < npairs;
    const int L = pv.lmax - m * pv.mres + 1;
    const int nseg = (L + kSeedSeg - 1) / kSeedSeg;
    const long col = col_of_mres(pv.lmax, m, pv.mres);
    const double x = in ? pv.x[p] : 0.0;
    double y1 = 0.0, y2 = in ? pv.pmm[(size_t)m * npairs + p] : 0.0;
    int k = in ? pv.pmmk[(size_t)m * npairs + p] : 0;
    int first = thr > 0.0 ? nseg : 0, kept = nseg;
    constexpr int kOne = 0x3ff00000, kStep = Scale<double>::S << 20;   // high words of 1 and of a step of k
    const int hthr = __double2hiint(thr), hkeep = seeds32 ? kOne + kLeast32 * (1 << 20) : kOne - kStep;
    for (int s = 0; s < nseg && in; ++s) {
        const size_t o = (segoff[m] + s) * npairs + p;
        const double b1 = y1, b2 = y2;   // the state entering the segment
        const int bk = k;
        int top = INT_MIN;   // high word of the segment's largest |P|, k steps taken off
        if (seeds64) {
            const int h = hseg[segoff[m] + s];
            seeds64[o] = make_double2(scalbn(y1, h), scalbn(y2, h));
            seeds64k[o] = k;
        }
        const int n1 = min(kSeedSeg, L - kSeedSeg * s);
        for (int i = 0; i < n1; ++i) {
            const double2 ab = pv.ab[col + kSeedSeg * s + i];
            const double yn = fma(ab.x * x, y1, ab.y * y2);
            y2 = y1;
            y1 = yn;
            int hi = __double2hiint(yn) & 0x7fffffff;
            if (k > 0 && hi >= kOne) {
                y1 *= 0x1p-240;
                y2 *= 0x1p-240;
                k -= 1;
                hi -= kStep;
            }
            top = max(top, hi - min(k, 3) * kStep);   // below 2^-700 all the same
        }
        if (s < first && top >= hthr) first = s;
        if (s < kept && top >= hkeep) kept = s;
        if (seeds32) seeds32[o] = fp32_state(b1, b2, bk, (top >> 20) - 1023);
    }
    if (in) live[(size_t)m * npairs + p] = (unsigned short)first;
    first = __reduce_min_sync(kFull, in ? first : 0xffff);
    kept = __reduce_min_sync(kFull, in ? kept : 0xffff);
    if ((threadIdx.x & 31) == 0 && in) {   // the group's first pair
        const size_t g = (size_t)m * groups_of(npairs) + (p >> 5);
        glive[g] = (unsigned short)first;
        glive_vec[g] = (unsigned short)kept;
    }
}

}  // namespace

cudaError_t launch_build_restarts(const PlanView<double> &pv, const unsigned long long *segoff, float4 *seeds32,
                                  double2 *seeds64, int *seeds64k, const int *hseg, unsigned short *live,
                                  unsigned short *glive, unsigned short *glive_vec, double thr, cudaStream_t st)
{
    dim3 grid((unsigned)((pv.npairs + 127) / 128), (unsigned)(pv.mmax + 1));
    k_build_restarts<<<grid, 128, 0, st>>>(pv, segoff, seeds32, seeds64, seeds64k, hseg, live, glive, glive_vec,
                                          thr);
    return cudaGetLastError();
}

}  // namespace sht
