// Augmented pattern: the experimental effects that synthetic training patterns
// for ML models carry (Sec. 1: peak broadening, noise, preferred orientation),
// applied on the GPU to the structure factors of the pattern path.
//
//   y_k = sum_g 2 I_g P_g PV(t_k - 2theta_g)   (Friedel-unique g; g and -g share I, P, 2theta)
//   P_g = (r^2 c + (1 - c) / r)^(-3/2),  c = cos^2 of the angle between g and n (metric G*)
//   PV(u) = eta (2 / (pi w)) / (1 + x^2) + (1 - eta) (2 / w) sqrt(ln 2 / pi) 2^(-x^2),  x = 2 u / w
//   then y_k += sigma sqrt(max(y_k, 0)) z_k.
//
// The structures come in order of their reflection count, largest first (aorder).
// k_aug_sum gives each warp 256 grid points of one structure (kAugPts
// consecutive points per thread) and streams all of the structure's reflections
// through shared memory, turning each into a record as it is staged: its grid
// cell b, the offset d of 2theta within the cell scaled by s = 2 dt / w, and the
// Lorentzian and Gaussian amplitudes. The Lorentzian has no window, but beyond
// kAugNear points from the middle of the warp's points a reflection's Lorentzian is
// smooth over them: those reflections are summed at kAugNodes of the points only
// (the Chebyshev-Lobatto points of the interval, rounded to the grid) and the sum is interpolated to all
// 256 by its polynomial through the nodes. At the least distance that errs by 7e-8 of the Lorentzian at the worst
// point, whatever the width (the poles of a Lorentzian lie at its 2theta, half a width off the real axis), about an
// FP32 rounding, and by rho^-16, rho = r + sqrt(r^2 - 1), r = distance / 127.5, farther out. The Gaussian and the near
// Lorentzians (an eighth of the reflections on 4096 points) are evaluated at every point; the Gaussian only for the reflections that reach
// the warp's points with x^2 < 40.
// What bounds it: instruction issue and the reciprocals, 2.2 instructions a clock (the CTAs also wait at the barriers
// around the staging): per reflection and warp about 2.5 instructions for a far one, 36 for a near Lorentzian and 30 for
// a Gaussian. 1024 cells of 1 to 64 atoms, 4096 points: 755 us with every (point, reflection) pair evaluated by
// itself, 275 us now; summing the tails once per node instead of in every point's long sum also took the error of the
// patterns from 4.6e-6 to 2e-7 of their norm.
//
// Precision: x = (k - b) s - d s with k - b an exact integer in FP32 (|k|, |b| <
// 2^22); for s <= 1 the points after a thread's first take x + j s (absolute
// error a few ulp of kAugPts s there); sums are FP32.
#include <cmath>

#include "xrd_internal.cuh"
#include "xrd_launch.h"

namespace xrd {

constexpr int kAugPts = 8;                       // consecutive grid points per thread
constexpr int kAugBlock = 32 * kAugPts;          // points of a warp
constexpr int kAugNodes = 16;                    // of them, the interpolation's
constexpr float kAugNear = 256.f;                // grid points from the warp's middle within which every point is summed
// Up to this many reflections of a structure are summed at every point, in their order: sorting them and weighting the
// nodes cost more (100 000 cells of a few reflections on 500 points 1.66 ms a call, now 1.32; 50 000 of about 40 on 128
// points 1.09, now 0.82).
constexpr int kAugFew = 64;

__device__ __forceinline__ float rcp_approx(float x)
{
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Per-structure constants of the profile sum (all zero for a structure that is
// invalid or has invalid effect parameters: no reflections, a zero row).
struct AugStruct {
    int n;             // reflections summed
    int valid, lor, gau, po;
    float sc;          // 2 dt / fwhm
    float cl, cg;      // Lorentzian and Gaussian prefactors of the area-normalised profile
    float m0, m1, m2;  // G* n / |n| (|n| in the metric G*): g.n / |n| = h m0 + k m1 + l m2
    float r;           // March-Dollase r
    float sig;         // noise scale
};

// Validates the effect parameters of structure s (every comparison is false
// for NaN, so NaN parameters fail). bad_params: the structure itself is valid
// but its parameters are not.
__device__ AugStruct aug_struct(const AugArgs& a, int s, bool& bad_params)
{
    AugStruct c{};
    const bool geo_ok = !*a.abort_flag && a.geo[s].status == XRD_OK;
    const double w = a.fwhm[s], eta = a.eta[s];
    const double sc = 2.0 * a.dt / w;
    bool ok = w > 0.0 && w <= 1e6 && sc <= 1e6 && eta >= 0.0 && eta <= 1.0;
    double M0 = 0.0, M1 = 0.0, M2 = 0.0, nn = 1.0, R = 1.0, sig = 0.0;
    if (a.po_dir && geo_ok) {
        const double* n = a.po_dir + 3 * (int64_t)s;
        const double* g = a.geo[s].gs;
        R = a.po_r[s];
        M0 = g[0] * n[0] + g[3] * n[1] + g[4] * n[2];
        M1 = g[3] * n[0] + g[1] * n[1] + g[5] * n[2];
        M2 = g[4] * n[0] + g[5] * n[1] + g[2] * n[2];
        nn = n[0] * M0 + n[1] * M1 + n[2] * M2;
        ok = ok && R >= 1e-6 && R <= 1e6 && nn > 0.0 && nn < INFINITY && fabs(M0) < INFINITY &&
             fabs(M1) < INFINITY && fabs(M2) < INFINITY;
    }
    if (a.noise_z) {
        sig = a.noise_sigma[s];
        ok = ok && sig >= 0.0 && sig < INFINITY;
    }
    bad_params = geo_ok && !ok;
    if (!(geo_ok && ok)) return c;
    c.n = (int)(a.refl_off[s + 1] - a.refl_off[s]);
    c.valid = 1;
    c.lor = eta > 0.0;
    c.gau = eta < 1.0;
    c.sc = (float)sc;
    c.cl = (float)(eta * 2.0 / (kPi * w));
    c.cg = (float)((1.0 - eta) * (2.0 / w) * sqrt(log(2.0) / kPi));
    c.po = a.po_dir != nullptr;
    const double inv = 1.0 / sqrt(nn);
    c.m0 = (float)(M0 * inv);
    c.m1 = (float)(M1 * inv);
    c.m2 = (float)(M2 * inv);
    c.r = (float)R;
    c.sig = (float)sig;
    return c;
}

// Record of reflection j: (-b, -d s, Lorentzian amplitude, Gaussian amplitude).
__device__ __forceinline__ float4 aug_record(const AugArgs& a, const AugStruct& c, int64_t j)
{
    const double q = a.q[j];
    const double T = two_theta_q(q, a.l2h, a.l2l, a.ttab);
    const double pos = (T - a.t0) * a.inv_dt;
    const double fb = floor(pos);
    float P = 1.f;
    if (c.po) {
        const uint32_t key = a.key[j];
        const float gn = fmaf((float)hkl_h(key), c.m0, fmaf((float)hkl_k(key), c.m1, (float)hkl_l(key) * c.m2));
        const float c2 = fminf(gn * gn / d2f_pos(q), 1.f);
        const float t = fmaf(c.r * c.r, c2, (1.f - c2) / c.r);
        P = 1.f / (t * sqrtf(t));
    }
    const float A = 2.f * a.Ig[j] * P;
    return make_float4(-(float)(int)fb, -(float)((pos - fb) * (double)c.sc), A * c.cl, A * c.cg);
}

// Lorentzian part of one reflection at a thread's kAugPts consecutive
// points, two points to a packed FP32 operation. x at the thread's
// first point is exact up to rounding ((k - b) is an exact integer in FP32).
// EXACT computes every point the same way; otherwise x_j = x_0 + j s in one fma
// (absolute error a few ulp of kAugPts s: used for s <= 1, i.e. fwhm >= 2 dt).
// acc[j] holds points 2 j + 1 and 2 j, in this order.
template <bool EXACT>
__device__ __forceinline__ void aug_lorentz(const float4 R, float kf, float sc, float2 (&acc)[kAugPts / 2])
{
    // R = (-b, -d s, Lorentzian amplitude, Gaussian amplitude)
    const float m0 = kf + R.x;
    const float2 s2 = make_float2(sc, sc), one = make_float2(1.f, 1.f);
    const float x0 = fmaf(m0, sc, R.y);
    // one reciprocal per pair of points: 1/d0 = d1 / (d0 d1). d <= 1 + 2^86 (2^23 grid steps of at most 1e6 in x): where
    // d0 d1 overflows both terms are below 2^-42 of the reflection's peak, and both become 0
#pragma unroll
    for (int j = 0; j < kAugPts; j += 2) {
        const float2 x = EXACT ? __ffma2_rn(make_float2(m0 + (float)j, m0 + (float)(j + 1)), s2, make_float2(R.y, R.y))
                               : __ffma2_rn(make_float2((float)j, (float)(j + 1)), s2, make_float2(x0, x0));
        const float2 d = __ffma2_rn(x, x, one);
        const float r = R.z * rcp_approx(d.x * d.y);
        acc[j / 2] = __ffma2_rn(d, make_float2(r, r), acc[j / 2]);
    }
}

// Gaussian part of one reflection at a thread's points
__device__ __forceinline__ void aug_gauss(const float4 R, float kf, float sc, float2 (&acc)[kAugPts / 2])
{
    const float m0 = kf + R.x;
#pragma unroll
    for (int j = 0; j < kAugPts; j += 2) {
        const float2 x = __ffma2_rn(make_float2(m0 + (float)(j + 1), m0 + (float)j), make_float2(sc, sc), make_float2(R.y, R.y));
        const float2 x2 = __fmul2_rn(x, x);
        acc[j / 2] = __ffma2_rn(make_float2(R.w, R.w), make_float2(ex2_approx(-x2.x), ex2_approx(-x2.y)), acc[j / 2]);
    }
}

// The interpolation's nodes, as offsets from a warp's first point: Chebyshev-Lobatto points of [0, 255], rounded.
static __constant__ int c_aug_node[kAugNodes] = {0, 3, 11, 24, 42, 64, 88, 114, 141, 167, 191, 213, 231, 244, 252, 255};
static __device__ float4 g_aug_w[kAugBlock][kAugNodes / 4];  // weight of each node's sum at each point

// Lagrange's basis on the nodes, in FP64: thread j of block k the weight of node j at point k
__global__ void k_aug_init()
{
    const int k = blockIdx.x, j = threadIdx.x;
    double num = 1.0, den = 1.0;
    for (int i = 0; i < kAugNodes; i++)
        if (i != j) {
            num *= (double)(k - c_aug_node[i]);
            den *= (double)(c_aug_node[j] - c_aug_node[i]);
        }
    ((float*)g_aug_w[k])[j] = (float)(num / den);
}

void init_aug_tables(cudaStream_t st) { k_aug_init<<<kAugBlock, kAugNodes, 0, st>>>(); }

// Staging order: the reflections of a chunk by the half block (128 points) that holds their 2theta, in the CTA's
// 2 WARPS half blocks, one more on either side and the two outer rests, by a stable counting sort. The half blocks
// of the reflections within kAugNear of a warp's middle are then four in a row: the near reflections are one range of
// the chunk and the far ones the two ranges beside it, with no test per reflection.
template <int WARPS>
struct AugStage {
    static constexpr int kThreads = 32 * WARPS, kChunk = 2 * kThreads, kGroups = kChunk / 32, kBins = 2 * WARPS + 4;
    float4 rec[kChunk];
    float2 b[kChunk / 2], ds[kChunk / 2], al[kChunk / 2];  // the far sum's operands, two reflections a load
    int cnt[kGroups][kBins + 1];  // of each 32 reflections, per bin; then the place of their first
    int start[kBins + 1];
    float4 node[WARPS][kAugNodes / 4];
    AugStruct cs;
};

// Resident warps: 32 per SM (48 would spill registers).
template <int WARPS>
__global__ void __launch_bounds__(32 * WARPS, 32 / WARPS) k_aug_sum(const AugArgs a, int nblk)
{
    pdl_enter();
    using S = AugStage<WARPS>;
    __shared__ S sh;
    const int ib = blockIdx.x / nblk;
    const int s = a.aorder[ib];
    const int k0 = (blockIdx.x - ib * nblk) * WARPS * kAugBlock;
    if (threadIdx.x == 0) {
        bool bad;
        sh.cs = aug_struct(a, s, bad);
        if (bad && k0 == 0) {  // flagged once, by the structure's first CTA
            a.status[s] = XRD_EINVAL;
            atomicAdd((unsigned long long*)&a.totals[3], 1ull);
        }
    }
    __syncthreads();
    const AugStruct& c = sh.cs;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, half = lane >> 4;
    const int kw = k0 + kAugBlock * warp;   // this warp's first grid point
    const int kt = kw + kAugPts * lane;     // this thread's first grid point
    const float kf = (float)kt, sc = c.sc;
    const bool lor = c.lor, gau = c.gau;
    float2 acc[kAugPts / 2];
#pragma unroll
    for (int j = 0; j < kAugPts / 2; j++) acc[j] = make_float2(0.f, 0.f);
    // none of the warp's points is within x^2 < 40 when |x| at their middle exceeds half their span in x plus sqrt(40)
    // (with margin); where that can be beyond kAugNear the Gaussians of the whole chunk are tested
    const float kc = (float)kw + 0.5f * (float)(kAugBlock - 1);
    const float reach = fmaf(0.5f * (float)(kAugBlock - 1), sc, 6.5f) * 1.0001f;
    const bool wide_gauss = reach >= (kAugNear - 2.f) * sc;
    const float knode = (float)(kw + c_aug_node[lane & 15]);  // the two halves of the warp take two reflections each at a time
    const float2 kn2 = make_float2(knode, knode), sc2 = make_float2(sc, sc), one = make_float2(1.f, 1.f);
    float2 far = make_float2(0.f, 0.f);
    const int64_t base = c.n ? a.refl_off[s] : 0;
    // Lorentzians of [n0, n1), Gaussians of [g0, g1). Four reflections of the first loop in flight: one after another, short
    // grids, most of whose reflections are near ones, took longer than without any far sums (64 small cells on 257 points
    // 606 us a call, 580 without; now 536).
    auto near_sums = [&](int n0, int n1, int g0, int g1) {
        if (lor) {
            if (sc <= 1.f)
#pragma unroll 4
                for (int i = n0; i < n1; i++) aug_lorentz<false>(sh.rec[i], kf, sc, acc);
            else
#pragma unroll 4
                for (int i = n0; i < n1; i++) aug_lorentz<true>(sh.rec[i], kf, sc, acc);
        }
        if (gau)
            for (int i0 = g0; i0 < g1; i0 += 32) {
                const int i = min(i0 + lane, g1 - 1);
                unsigned b = __ballot_sync(0xffffffffu, i0 + lane < g1 && fabsf(fmaf(kc + sh.rec[i].x, sc, sh.rec[i].y)) < reach);
                for (; b; b &= b - 1) aug_gauss(sh.rec[i0 + __ffs(b) - 1], kf, sc, acc);
            }
    };
    const bool few = c.n <= kAugFew;
    if (few && c.n > 0) {
        static_assert(kAugFew <= S::kThreads, "a reflection a thread");
        if ((int)threadIdx.x < c.n) sh.rec[threadIdx.x] = aug_record(a, c, base + threadIdx.x);
        __syncthreads();
        if (kw < a.n_pts) near_sums(0, c.n, 0, c.n);
    }
    for (int c0 = 0; !few && c0 < c.n; c0 += S::kChunk) {
        const int m = min((int)S::kChunk, c.n - c0);
        float4 R[2];
        int bin[2], rank[2];
        __syncthreads();  // the previous chunk is done with
        for (int i = threadIdx.x; i < S::kGroups * (S::kBins + 1); i += S::kThreads) (&sh.cnt[0][0])[i] = 0;
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const int g = warp + u * WARPS, i = 32 * g + lane;
            R[u] = make_float4(0.f, 0.f, 0.f, 0.f);
            bin[u] = S::kBins;  // past the end: no reflection
            if (i < m) {
                R[u] = aug_record(a, c, base + c0 + i);
                bin[u] = min(max((((int)-R[u].x - k0) >> 7) + 2, 0), S::kBins - 1);
            }
            const unsigned peers = __match_any_sync(0xffffffffu, bin[u]);
            rank[u] = __popc(peers & ((1u << lane) - 1u));
            if (rank[u] == 0) sh.cnt[g][bin[u]] = __popc(peers);
        }
        __syncthreads();
        for (int b = threadIdx.x; b <= S::kBins; b += S::kThreads) {  // places within the bin
            int run = 0;
            for (int g = 0; g < S::kGroups; g++) {
                const int v = sh.cnt[g][b];
                sh.cnt[g][b] = run;
                run += v;
            }
            sh.start[b] = run;
        }
        __syncthreads();
        if (warp == 0) {  // bins in their order
            int carry = 0;
            for (int b0 = 0; b0 <= S::kBins; b0 += 32) {
                const int v = b0 + lane <= S::kBins ? sh.start[b0 + lane] : 0;
                const int inc = warp_incl_scan(v);
                if (b0 + lane <= S::kBins) sh.start[b0 + lane] = carry + inc - v;
                carry += __shfl_sync(0xffffffffu, inc, 31);
            }
        }
        __syncthreads();
#pragma unroll
        for (int u = 0; u < 2; u++) {
            const int at = sh.start[bin[u]] + sh.cnt[warp + u * WARPS][bin[u]] + rank[u];
            sh.rec[at] = R[u];
            ((float*)sh.b)[at] = R[u].x;
            ((float*)sh.ds)[at] = R[u].y;
            ((float*)sh.al)[at] = R[u].z;
        }
        __syncthreads();
        if (kw >= a.n_pts) continue;  // uniform in the warp
        const int n0 = sh.start[2 * warp + 1], n1 = sh.start[2 * warp + 5];  // the near reflections
        if (lor) {
            auto far_pair = [&](int i, float2 A) {  // reflections 2 i and 2 i + 1 at this lane's node
                const float2 x = __ffma2_rn(__fadd2_rn(kn2, sh.b[i]), sc2, sh.ds[i]);
                const float2 d = __ffma2_rn(x, x, one);
                far = __ffma2_rn(A, make_float2(rcp_approx(d.x), rcp_approx(d.y)), far);
            };
            auto far_range = [&](int lo, int hi) {  // [lo, hi), the halves of the warp on alternate pairs
                const int p0 = lo >> 1, p1 = (hi + 1) >> 1;  // pairs; the first and the last may reach past the range
                for (int i = p0 + half; i < p1; i += 2) {
                    float2 A = sh.al[i];
                    if (2 * i < lo) A.x = 0.f;
                    if (2 * i + 1 >= hi) A.y = 0.f;
                    far_pair(i, A);
                }
            };
            far_range(0, n0);
            far_range(n1, m);
        }
        near_sums(n0, n1, wide_gauss ? 0 : n0, wide_gauss ? m : n1);
    }
    float f = far.x + far.y;
    f += __shfl_xor_sync(0xffffffffu, f, 16);
    if (lane < kAugNodes) ((float*)sh.node[warp])[lane] = f;
    __syncwarp();
    if (kw >= a.n_pts) return;
    const bool valid = c.valid, noise = valid && a.noise_z != nullptr;
    float* __restrict__ yo = a.y + (int64_t)s * a.n_pts;
    const float* __restrict__ zo = noise ? a.noise_z + (int64_t)s * a.n_pts : nullptr;
#pragma unroll
    for (int j = 0; j < kAugPts; j++) {
        const int k = kt + j;
        if (k >= a.n_pts) break;
        float v = j & 1 ? acc[j / 2].x : acc[j / 2].y;
        if (lor && !few) {
            float f = 0.f;
#pragma unroll
            for (int q = 0; q < kAugNodes / 4; q++) {
                const float4 w = g_aug_w[kAugPts * lane + j][q], n = sh.node[warp][q];
                f = fmaf(w.x, n.x, fmaf(w.y, n.y, fmaf(w.z, n.z, fmaf(w.w, n.w, f))));
            }
            v += f;
        }
        if (noise) v = fmaf(c.sig * sqrtf(fmaxf(v, 0.f)), zo[k], v);
        yo[k] = valid ? v : 0.f;
    }
}

// CTAs of 8 warps (2048 points share a staging), or of 4 for grids of up to 1024 points. The width sets the chunk and so
// the order of the FP32 sums: it follows the grid alone, and a structure's pattern is the same bits in any batch. (Narrow
// CTAs for small batches too, to fill the SMs, gave nothing: 24 small cells on 4096 points 193 us, 186 with wide ones, 4
// cells 97 both.) 16 warps a CTA took the same time on 4096 points.
void launch_aug(const AugArgs& a, cudaStream_t st)
{
    if (a.n_struct <= 0) return;
    if (a.n_pts > 4 * kAugBlock) {
        const int nblk = (a.n_pts + 8 * kAugBlock - 1) / (8 * kAugBlock);
        launch_pdl(k_aug_sum<8>, (unsigned)((int64_t)a.n_struct * nblk), 256, 0, st, a, nblk);
    } else {
        launch_pdl(k_aug_sum<4>, (unsigned)a.n_struct, 128, 0, st, a, 1);
    }
}

}  // namespace xrd
