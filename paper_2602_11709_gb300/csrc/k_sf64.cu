// Steps S2-S3 in FP64: structure factor and intensity of the XRD_FP64 variant.
//
// Sec. 2: F(g) = sum_j occ_j f_j(s) exp(-B_j s^2) exp(2 pi i g.x_j), I = |F|^2 LP (see k_sf.cu for the formulas).
//
// What bounds it: this part issues 1.7 FP64 lane operations per clock and SM against 64 to 128 integer ones, so
// a term written with the library's sincospi and exp (about 110 FP64 operations with its share of f(s)) leaves
// every other unit idle. Here the phase is exact in 64-bit fixed point, sin, cos and the five exponentials
// of a term are formed in integers (xrd_fx.cuh, accurate to the last bit of a double), f(s) is summed in fixed
// point, and FP64 keeps the products and the sums: four operations per term, plus two per element run.
// Measured, 1024 cells of 1 to 64 atoms (1.03 M reflections, 35 M terms): 7.27 ms with the library's functions, 0.88 ms
// here (ALU pipe 53 %, FP64 pipe 40 %, 2.4 instructions a clock); the whole call 7.40 -> 1.00 ms.
#include "xrd_fx.cuh"
#include "xrd_internal.cuh"
#include "xrd_launch.h"

namespace xrd {

constexpr int kSf64Warps = 4;
constexpr int kSf64Chunk = 32;  // atoms staged per warp at a time

static __device__ uint64_t g_fx_exp[kFxExpN];
static __device__ ulonglong2 g_fx_sc[kFxScN + 1];

// ---- tables, formed once per handle in double-double (error-free sums and FMA products) ----

struct HD {
    double h, l;
};
__device__ __forceinline__ HD hd_fast(double h, double l)
{
    const double s = __dadd_rn(h, l);
    return HD{s, __dsub_rn(l, __dsub_rn(s, h))};
}
__device__ __forceinline__ HD hd_add(HD a, HD b)
{
    const double s = __dadd_rn(a.h, b.h), bb = __dsub_rn(s, a.h);
    const double e = __dadd_rn(__dsub_rn(a.h, __dsub_rn(s, bb)), __dsub_rn(b.h, bb));
    return hd_fast(s, __dadd_rn(e, __dadd_rn(a.l, b.l)));
}
__device__ __forceinline__ HD hd_mul(HD a, HD b)
{
    const double p = __dmul_rn(a.h, b.h);
    return hd_fast(p, __dadd_rn(__fma_rn(a.h, b.h, -p), __fma_rn(a.h, b.l, __dmul_rn(a.l, b.h))));
}
// a >= 0 in units of 2^-bits, rounded
__device__ uint64_t hd_fixed(HD a, int bits)
{
    const double sc = scalbn(1.0, bits), v = a.h * sc, f = floor(v);
    return (uint64_t)f + (uint64_t)__double2ll_rn((v - f) + a.l * sc);
}

__global__ void k_fx_init()
{
    constexpr int kTerms = 30;
    __shared__ HD inv[kTerms + 1];  // 1 / k
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (threadIdx.x < kTerms) {
        const double k = threadIdx.x + 1.0, h = __ddiv_rn(1.0, k);
        inv[threadIdx.x + 1] = HD{h, __ddiv_rn(__fma_rn(-h, k, 1.0), k)};
    }
    __syncthreads();
    if (i < kFxExpN) {  // 2^(-i / kFxExpN) by the series of exp
        const HD x = hd_mul(HD{0.6931471805599453, 2.3190468138462996e-17}, HD{-i / (double)kFxExpN, 0.0});
        HD t{1.0, 0.0}, s = t;
        for (int k = 1; k <= 24; k++) s = hd_add(s, t = hd_mul(hd_mul(t, x), inv[k]));
        g_fx_exp[i] = i ? hd_fixed(s, 64) : ~0ull;
        return;
    }
    const int j = i - kFxExpN;
    if (j > kFxScN) return;
    const HD x = hd_mul(HD{1.5707963267948966, 6.123233995736766e-17}, HD{j / (double)kFxScN, 0.0});
    HD t{1.0, 0.0}, c = t, s{0.0, 0.0};
    for (int k = 1; k <= kTerms; k++) {
        t = hd_mul(hd_mul(t, x), inv[k]);
        const HD v = k & 2 ? HD{-t.h, -t.l} : t;
        if (k & 1) s = hd_add(s, v);
        else c = hd_add(c, v);
    }
    g_fx_sc[j] = make_ulonglong2(j == kFxScN ? 0ull : hd_fixed(c, 62), hd_fixed(s, 62));
}

void init_fx_tables(cudaStream_t st) { k_fx_init<<<(kFxExpN + kFxScN + 1 + 31) / 32, 32, 0, st>>>(); }

// ---- f(s) of one element: Z - 41.78214 s^2 sum_i a_i exp(-b_i s^2) ----

// Coefficients of one element in fixed point (fx_exp_sum). slow: one of them is outside the fixed-point form (negative
// or huge b, denormal a, not finite); f is then formed in FP64 with the library's exp.
struct CoefX {
    uint64_t bm[4];
    uint64_t am[4];
    int16_t be[4], ae[4];
    int slow, pad;
};

__device__ void coefx_of(const double* __restrict__ c, CoefX& o)
{
    bool ok = true;
    for (int i = 0; i < 4; i++) {
        const double a = c[2 * i];
        const FxNum b = fx_log2e(c[2 * i + 1]);
        int e;
        o.am[i] = fx_signed(a, e);
        o.ae[i] = (int16_t)e;
        o.bm[i] = b.m;
        o.be[i] = (int16_t)(b.e == kFxSlow ? 0 : b.e);
        ok = ok && b.e != kFxSlow && (a == 0.0 || (fabs(a) >= 0x1p-300 && fabs(a) <= 0x1p300));
    }
    o.slow = !ok;
    o.pad = 0;
}

__device__ __noinline__ double f64_slow(const double* __restrict__ c, int z, double s2)
{
    const double sum = c[0] * exp(-c[1] * s2) + c[2] * exp(-c[3] * s2) + c[4] * exp(-c[5] * s2) +
                       c[6] * exp(-c[7] * s2);
    return (double)z - kFScale * s2 * sum;
}

__device__ __noinline__ double dw64_slow(double B, double s2) { return exp(-B * s2); }

__device__ __forceinline__ double f64_of(const CoefX& c, double zf, double s2, FxNum S, const uint64_t* __restrict__ ex)
{
    return fma(-kFScale * s2, fx_exp_sum(c.am, c.ae, c.bm, c.be, S, ex), zf);
}

// h x + k y + l z mod 1 in 64-bit fixed point, exact for the record's coordinates
__device__ __forceinline__ uint64_t phase64(const AtomX& a, int h, int k, int l)
{
    const int64_t lo = (int64_t)h * a.lo[0] + (int64_t)k * a.lo[1] + (int64_t)l * a.lo[2];
    const uint32_t hi = (uint32_t)h * a.hi[0] + (uint32_t)k * a.hi[1] + (uint32_t)l * a.hi[2];
    return (uint64_t)lo + ((uint64_t)hi << 32);
}

// Persistent CTAs; every warp takes tiles of 32 RB reflections (RB per lane, 32 apart) from the queue in
// largest-first order and walks the structure's element-sorted atoms, staged 32 at a time.
template <int RB>
__global__ void __launch_bounds__(32 * kSf64Warps, 5) k_sf64(const SfArgs a)
{
    pdl_enter();
    __shared__ uint64_t ex[kFxExpN];
    __shared__ ulonglong2 sc[kFxScN + 1];
    __shared__ AtomX sat[kSf64Warps][kSf64Chunk];
    extern __shared__ __align__(16) unsigned char coef_raw[];
    CoefX* const scoef = (CoefX*)coef_raw;  // [zmax + 1]
    if (*a.abort_flag) return;
    const int ntiles = a.tile_off[a.n_struct];
    if ((int)blockIdx.x >= ntiles) return;  // the CTAs before this one already have a tile each
    for (int i = threadIdx.x; i < kFxExpN; i += blockDim.x) ex[i] = g_fx_exp[i];
    for (int i = threadIdx.x; i <= kFxScN; i += blockDim.x) sc[i] = g_fx_sc[i];
    for (int z = threadIdx.x; z <= a.zmax; z += blockDim.x) coefx_of(a.coef + 8 * z, scoef[z]);
    __syncthreads();
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (;;) {
        int t = 0;
        if (lane == 0) t = atomicAdd(a.tile_counter, 1);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= ntiles) break;
        const int2 e = a.tile_tab[t];
        const int64_t rbase = a.refl_off[e.x], re = a.refl_off[e.x + 1];
        const int64_t j0 = a.atom_off[e.x], j1 = a.atom_off[e.x + 1];
#pragma unroll 1
        for (int i = 0; i < RB; i++) {
            if (rbase + e.y + 32 * i >= re) break;  // uniform
            const int64_t r = rbase + e.y + 32 * i + lane;
            const bool act = r < re;
            const int64_t rr = act ? r : rbase;
            const uint32_t key = a.key[rr];
            const double q = a.q[rr], s2 = q * 0.25;
            const FxNum S = fx_num(s2);
            const int h = hkl_h(key), k = hkl_k(key), l = hkl_l(key);
            double Fr = 0.0, Fi = 0.0, f = 0.0;
            int zc = -1;
            for (int64_t c0 = j0; c0 < j1; c0 += kSf64Chunk) {
                const int nc = (int)min((int64_t)kSf64Chunk, j1 - c0);
                __syncwarp();
                if (lane < nc) sat[w][lane] = a.atomx[c0 + lane];
                __syncwarp();
#pragma unroll 1
                for (int jj = 0; jj < nc; jj++) {
                    const AtomX& at = sat[w][jj];
                    const int z = at.z;
                    if (z != zc) {  // uniform: every lane walks the same element-sorted list
                        zc = z;
                        const CoefX& c = scoef[z];
                        f = c.slow ? f64_slow(a.coef + 8 * z, z, s2) : f64_of(c, (double)z, s2, S, ex);
                    }
                    int64_t ci, si;
                    fx_sincos(phase64(at, h, k, l), sc, ci, si);
                    double dw;
                    if (at.be != kFxSlow) {  // uniform
                        int n;
                        const uint64_t m = fx_exp2_neg(at.bm, at.be, S.m, S.e, ex, n);
                        dw = fx_exp_double(m, n);
                    } else {
                        dw = dw64_slow(fx_as_double(at.bm), s2);
                    }
                    const double wt = at.occ * f * dw;
                    Fr = fma(wt, fx_to_double<62>(ci), Fr);
                    Fi = fma(wt, fx_to_double<62>(si), Fi);
                }
            }
            if (act) {
                const double X = (a.lambda * a.lambda * 0.25) * q;  // sin^2 theta
                const double c2 = 1.0 - 2.0 * X;                     // cos 2theta
                const double lp = (1.0 + c2 * c2) / (X * sqrt(fmax(1.0 - X, kCos90Sq)));
                a.I[r] = (Fr * Fr + Fi * Fi) * lp;
                if (a.F) a.F[r] = make_float2((float)Fr, (float)Fi);
            }
        }
    }
}

template <int RB>
static void launch_sf64_rb(const SfArgs& a, cudaStream_t st, bool pdl)
{
    const size_t smem = sizeof(CoefX) * (size_t)(a.zmax + 1);
    const int per_sm = resident_ctas((const void*)k_sf64<RB>, 32 * kSf64Warps, smem);
    if (pdl) launch_pdl(k_sf64<RB>, a.grid * per_sm, 32 * kSf64Warps, smem, st, a);
    else k_sf64<RB><<<a.grid * per_sm, 32 * kSf64Warps, smem, st>>>(a);
}

void launch_sf64(const SfArgs& a, cudaStream_t st, bool pdl)
{
    if (a.rb == 1) launch_sf64_rb<1>(a, st, pdl);
    else if (a.rb == 2) launch_sf64_rb<2>(a, st, pdl);
    else launch_sf64_rb<4>(a, st, pdl);
}

}  // namespace xrd
