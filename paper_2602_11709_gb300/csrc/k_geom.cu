// Steps S0-S1: per-structure geometry, atom packing and reflection enumeration.
//
// Sec. 2: the first step of the numerical core enumerates the reciprocal-lattice
// points that the wavelength and the 2-theta range can reach (a sphere in
// reciprocal space): every integer g = (h, k, l) != 0 with r_min <= |g| <= r_max, |g|^2 = h^T G* h.
// Friedel's law F(-g) = F(g)* makes g and -g identical in intensity, so only
// the half-space (first nonzero of h, k, l positive) is enumerated; every kept
// reflection stands for two.
//
// |g|^2 is evaluated in one fixed order with every product and sum rounded on
// its own (no fused multiply-add), so the set of reflections on the sphere
// boundary is decided exactly as a plain FP64 evaluation of the same order.
#include <algorithm>
#include <cmath>

#include "xrd_dd.cuh"
#include "xrd_fx.cuh"
#include "xrd_internal.cuh"
#include "xrd_launch.h"

namespace xrd {

__device__ __forceinline__ double cosd(double deg)
{
    // exact cosines at 90, 60 and 120 degrees; otherwise cos(deg * pi / 180)
    if (deg == 90.0) return 0.0;
    if (deg == 60.0) return 0.5;
    if (deg == 120.0) return -0.5;
    return cos(__dmul_rn(deg, kPi / 180.0));
}

// S0: reciprocal metric G* = G^-1 from the direct metric
// G = [[a^2, ab cos(gamma), ac cos(beta)], [., b^2, bc cos(alpha)], [., ., c^2]]
// by cofactors over the determinant, and the enumeration box |h| <= r_max a + 1.
// The part has little FP64 throughput. A small batch is latency-bound, so
// each structure takes LANES = 8 lanes: lanes 0-2 form the three cosines,
// every lane the cofactors and determinant (same operations, same order), lane
// j < 6 the element j of G* (one division each), lane 6 the box, status and
// hexagonal flag. A large batch is throughput-bound and takes one lane per
// structure (LANES = 1, no redundant work). Every value is rounded exactly as
// in a one-thread evaluation either way.
// Also zeroes the structure's largest-intensity slot (imax, written by the
// structure-factor pass) and writes its flag word (bit 0: hexagonal) when the
// pointers are given.
template <int LANES>
__device__ __forceinline__ void prep_thread(int t, const double* __restrict__ lattice, int n, double rmax,
                                            Geo* __restrict__ geo, unsigned* __restrict__ imax,
                                            int32_t* __restrict__ flags, const EnumParts& ep)
{
    const int s_raw = t / LANES, lane = t % LANES;
    const bool live = s_raw < n;
    if (LANES == 1 && !live) return;
    const int s = live ? s_raw : n - 1;  // lanes past the batch compute a copy and store nothing
    const double a = lattice[6 * s], b = lattice[6 * s + 1], c = lattice[6 * s + 2];
    const double al = lattice[6 * s + 3], be = lattice[6 * s + 4], ga = lattice[6 * s + 5];
    Geo& g = geo[s];
    const bool finite = isfinite(a) && isfinite(b) && isfinite(c) && isfinite(al) && isfinite(be) && isfinite(ga);
    bool ok = finite && a > 0.0 && b > 0.0 && c > 0.0;
    double ca, cb, cg;
    if (LANES == 1) {
        ca = ok ? cosd(al) : 0.0;
        cb = ok ? cosd(be) : 0.0;
        cg = ok ? cosd(ga) : 0.0;
    } else {
        const double cj = (ok && lane < 3) ? cosd(lane == 0 ? al : (lane == 1 ? be : ga)) : 0.0;
        ca = __shfl_sync(0xffffffffu, cj, 0, LANES);
        cb = __shfl_sync(0xffffffffu, cj, 1, LANES);
        cg = __shfl_sync(0xffffffffu, cj, 2, LANES);
    }
    // volume factor 1 - ca^2 - cb^2 - cg^2 + 2 ca cb cg, left to right
    double vf = __dsub_rn(1.0, __dmul_rn(ca, ca));
    vf = __dsub_rn(vf, __dmul_rn(cb, cb));
    vf = __dsub_rn(vf, __dmul_rn(cg, cg));
    vf = __dadd_rn(vf, __dmul_rn(__dmul_rn(__dmul_rn(2.0, ca), cb), cg));
    ok = ok && vf > 1e-6;
    const double G11 = __dmul_rn(a, a), G22 = __dmul_rn(b, b), G33 = __dmul_rn(c, c);
    const double G12 = __dmul_rn(__dmul_rn(a, b), cg);
    const double G13 = __dmul_rn(__dmul_rn(a, c), cb);
    const double G23 = __dmul_rn(__dmul_rn(b, c), ca);
    const double C11 = __dsub_rn(__dmul_rn(G22, G33), __dmul_rn(G23, G23));
    const double C12 = __dsub_rn(__dmul_rn(G13, G23), __dmul_rn(G12, G33));
    const double C13 = __dsub_rn(__dmul_rn(G12, G23), __dmul_rn(G13, G22));
    const double det = __dadd_rn(__dadd_rn(__dmul_rn(G11, C11), __dmul_rn(G12, C12)), __dmul_rn(G13, C13));
    if (!live) return;
#pragma unroll
    for (int j = (LANES == 1 ? 0 : lane); j < (LANES == 1 ? 7 : lane + 1); j++) {
        if (j < 6) {
            // element j of G* (stored as 11, 22, 33, 12, 13, 23)
            double Cj;
            switch (j) {
            case 0: Cj = C11; break;
            case 1: Cj = __dsub_rn(__dmul_rn(G11, G33), __dmul_rn(G13, G13)); break;
            case 2: Cj = __dsub_rn(__dmul_rn(G11, G22), __dmul_rn(G12, G12)); break;
            case 3: Cj = C12; break;
            case 4: Cj = C13; break;
            default: Cj = __dsub_rn(__dmul_rn(G12, G13), __dmul_rn(G11, G23)); break;
            }
            const double v = ok ? __ddiv_rn(Cj, det) : 0.0;
            g.gs[j] = v;
            const float v32 = ok ? __double2float_rn(v) : 0.f;
            g.gf[j] = v32;
            g.gl[j] = ok ? __double2float_rn(v - (double)v32) : 0.f;
        } else if (j == 6) {
            g.hex = fabs(al - 90.0) < 5.0 && fabs(be - 90.0) < 5.0 && fabs(ga - 120.0) < 5.0 && fabs(a - b) < 0.01;
            if (imax) imax[s] = 0u;
            if (flags) flags[s] = g.hex ? XRD_FLAG_HEXAGONAL : 0;
            int H = -1, K = -1, L = -1, st = XRD_EINVAL;
            if (ok) {
                H = (int)floor(__dmul_rn(rmax, a)) + 1;
                K = (int)floor(__dmul_rn(rmax, b)) + 1;
                L = (int)floor(__dmul_rn(rmax, c)) + 1;
                st = XRD_OK;
                if (H > kHklLimit || K > kHklLimit || L > kHklLimit) {
                    st = XRD_EINVAL;  // cell too large for the packed (h, k, l) key at this 2-theta range
                    H = K = L = -1;
                }
            }
            g.H = H;
            g.K = K;
            g.L = L;
            g.status = st;
            // the enumeration's parts of a structure with many columns (k_count, k_emit)
            int pbase = -1;
            const int ncol = H < 0 ? 0 : (K + 1) + H * (2 * K + 1);
            if (ncol > ep.cols) {
                const int np = (ncol + ep.cols - 1) / ep.cols;
                // 64 bits: up to 4088 parts a structure, room or not
                const long long b = (long long)atomicAdd(ep.ctr, (unsigned long long)np);
                const bool room = b <= ep.cap - np;
                if (room) pbase = (int)b;
                for (int i = 0; i < np && b + i < ep.cap; i++) ep.tab[b + i] = make_int2(room ? s : -1, i);
                if (room) {
                    ep.cnt[s] = 0;
                    if (ep.run_cnt) ep.run_cnt[s] = 0;
                }
            }
            g.pbase = pbase;
        }
    }
}

template <int LANES>
__global__ void k_prep(const double* __restrict__ lattice, int n, double rmax, Geo* __restrict__ geo,
                       unsigned* __restrict__ imax, int32_t* __restrict__ flags, const EnumParts ep)
{
    pdl_enter();
    prep_thread<LANES>(blockIdx.x * blockDim.x + threadIdx.x, lattice, n, rmax, geo, imax, flags, ep);
}

// 8 lanes per structure up to this many structures (latency-bound), one above (throughput-bound)
constexpr int kPrepWideMax = 8192;

// f(s) coefficients in the form the FP32 loops use (exp2 with the scale folded
// in) and, for the accurate re-evaluation, (a_i, b_i) as two floats each
// (cdd[4 z + i] = (a hi, a lo, b hi, b lo); skipped when cdd is null).
__device__ __forceinline__ void coef_block(const double* __restrict__ coef, int zmax, Coef32* __restrict__ c32,
                                           float4* __restrict__ cdd)
{
    for (int z = threadIdx.x; z <= zmax; z += blockDim.x) {
        Coef32 c;
        for (int i = 0; i < 4; i++) {
            const double av = coef[8 * z + 2 * i], bv = coef[8 * z + 2 * i + 1];
            c.a[i] = (float)(-kFScale * av);
            c.bl[i] = (float)(-bv * 1.4426950408889634);
            if (cdd) {
                const float ah = __double2float_rn(av), bh = __double2float_rn(bv);
                cdd[4 * z + i] = make_float4(ah, __double2float_rn(av - (double)ah), bh,
                                             __double2float_rn(bv - (double)bh));
            }
        }
        c32[z] = c;
    }
}

__global__ void k_coef(const double* __restrict__ coef, int zmax, Coef32* __restrict__ c32, float4* __restrict__ cdd)
{
    pdl_enter();
    coef_block(coef, zmax, c32, cdd);
}

// Validate and pack the atoms of one structure, sorted by element (stable:
// ties keep their input order) so that f(s) is evaluated once per element run.
constexpr int kAtomThreads = 128;
struct AtomShared {
    int off[kZmaxLimit + 1];
    int pos[kAtomThreads];
    int bad;
};
__device__ __forceinline__ void atoms_block(int s, AtomShared& sh, const int64_t* __restrict__ atom_off, int64_t n_atoms,
                                               const double* __restrict__ frac, const int16_t* __restrict__ Zin,
                                               const double* __restrict__ occ, const double* __restrict__ Bf, int zmax,
                                               Geo* __restrict__ geo, int set_geo, int* __restrict__ atom_bad,
                                               Atom32* __restrict__ a32, AtomX* __restrict__ ax,
                                               float2* __restrict__ astep, AtomR* __restrict__ ar,
                                               const float4* __restrict__ sctab)
{
    int* const off = sh.off;
    int64_t a0 = atom_off[s], na = atom_off[s + 1] - a0;
    const bool range_ok = a0 >= 0 && na >= 0 && atom_off[s + 1] <= n_atoms && na <= (1 << 30);
    if (!range_ok) { a0 = 0; na = 0; }
    for (int i = threadIdx.x; i <= kZmaxLimit; i += blockDim.x) off[i] = 0;
    if (threadIdx.x == 0) sh.bad = !range_ok;
    __syncthreads();
    for (int64_t i = threadIdx.x; i < na; i += blockDim.x) {
        const int z = Zin[a0 + i];
        const double x = frac[3 * (a0 + i)], y = frac[3 * (a0 + i) + 1], w = frac[3 * (a0 + i) + 2];
        const bool ok = z >= 0 && z <= zmax && isfinite(x) && isfinite(y) && isfinite(w) && occ[a0 + i] >= 0.0 &&
                        isfinite(occ[a0 + i]) &&
                        isfinite(Bf[a0 + i]) && fabs(x) < 262144.0 && fabs(y) < 262144.0 && fabs(w) < 262144.0;
        if (!ok) atomicOr(&sh.bad, 1);
        else atomicAdd(&off[z], 1);
    }
    __syncthreads();
    if (threadIdx.x == 0) atom_bad[s] = sh.bad;
    if (sh.bad) {
        // neutral records (weight 0, element 0) keep the structure-factor kernel's reads in bounds;
        // the structure reports XRD_EINVAL and gets no peaks
        if (threadIdx.x == 0 && set_geo) geo[s].status = XRD_EINVAL;
        for (int64_t i = threadIdx.x; i < na; i += blockDim.x) {
            Atom32 r{};
            r.lo = -INFINITY;
            r.src = (int)i;
            a32[a0 + i] = r;
            if (ax) ax[a0 + i] = AtomX{};
            if (astep) astep[a0 + i] = make_float2(1.f, 0.f);
            if (ar) {
                AtomR e{};
                ar[a0 + i] = e;
            }
        }
        return;
    }
    if (threadIdx.x < 32) {  // exclusive offset of each element's run: one warp, 8 elements a lane
        constexpr int per = (kZmaxLimit + 1) / 32;
        const int lane = threadIdx.x;
        int v[per], sum = 0;
#pragma unroll
        for (int k = 0; k < per; k++) {
            const int z = lane * per + k;
            v[k] = z <= zmax ? off[z] : 0;
            sum += v[k];
        }
        int run = warp_incl_scan(sum) - sum;
#pragma unroll
        for (int k = 0; k < per; k++) {
            const int z = lane * per + k;
            if (z <= zmax) off[z] = run;
            run += v[k];
        }
    }
    __syncthreads();
    // stable placement, one chunk of blockDim atoms at a time: the first warp ranks the chunk's atoms among those of
    // their element, 32 at a time, and advances the elements' offsets; then every thread packs its atom
    for (int64_t base = 0; base < na; base += blockDim.x) {
        const int64_t i = base + threadIdx.x;
        const int z = i < na ? (int)Zin[a0 + i] : -1;
        sh.pos[threadIdx.x] = z;
        __syncthreads();
        if (threadIdx.x < 32) {
            const int lane = threadIdx.x;
            for (int c = 0; c < (int)blockDim.x && base + c < na; c += 32) {
                const int zz = sh.pos[c + lane];
                const unsigned peers = __match_any_sync(0xffffffffu, zz);
                const int first = zz >= 0 ? off[zz] : 0;
                __syncwarp();
                if (zz >= 0 && lane == __ffs(peers) - 1) off[zz] = first + __popc(peers);
                __syncwarp();
                sh.pos[c + lane] = first + __popc(peers & ((1u << lane) - 1u));
            }
        }
        __syncthreads();
        if (i < na) {
            const int pos = sh.pos[threadIdx.x];
            const double x = frac[3 * (a0 + i)], y = frac[3 * (a0 + i) + 1], w = frac[3 * (a0 + i) + 2];
            const double o = occ[a0 + i], bb = Bf[a0 + i];
            Atom32 r;
            r.X = fix32(x);
            r.Y = fix32(y);
            r.Z = fix32(w);
            r.nb = (float)(-bb * 1.4426950408889634);
            r.lo = o == 1.0 ? 0.f : (o > 0.0 ? (float)log2(o) : -INFINITY);
            r.z = z;
            r.src = (int)i;
            r.zf = (float)z;
            a32[a0 + pos] = r;
            if (astep) {  // the l -> l + 1 step of the phase factor (runs), from the same fixed-point z:
                          // cos and sin of 2 pi z in double-float (FP32 operations), rounded to floats
                DD cz, sz;
                dd_sincos_turn((unsigned long long)r.Z << 32, sctab, cz, sz);
                astep[a0 + pos] = make_float2(cz.hi + cz.lo, sz.hi + sz.lo);
            }
            if (ax) {  // 64-bit fixed point with a signed low word, B log2(e) in fixed point
                AtomX d;
                const double v[3] = {x, y, w};
#pragma unroll
                for (int c = 0; c < 3; c++) {
                    const unsigned long long F = fix64(v[c]);
                    d.hi[c] = (uint32_t)((F + 0x80000000ull) >> 32);
                    d.lo[c] = (int32_t)(uint32_t)F;
                }
                const FxNum nb = fx_log2e(bb);
                d.bm = nb.e == kFxSlow ? fx_as_bits(bb) : nb.m;
                d.be = nb.e;
                d.z = z;
                d.occ = o;
                ax[a0 + pos] = d;
            }
            if (ar) {  // the accurate re-evaluation's record: 64-bit fixed point, two-float occ and B
                AtomR e;
                e.X = fix64(x);
                e.Y = fix64(y);
                e.Z = fix64(w);
                e.oh = __double2float_rn(o);
                e.ol = __double2float_rn(o - (double)e.oh);
                e.bh = __double2float_rn(bb);
                e.bl = __double2float_rn(bb - (double)e.bh);
                e.z = z;
                e.pad = 0;
                ar[a0 + pos] = e;
            }
        }
        __syncthreads();  // the positions are read before the next chunk's
    }
}

__global__ void __launch_bounds__(kAtomThreads) k_atoms(const int64_t* __restrict__ atom_off, int64_t n_atoms,
                                                        const double* __restrict__ frac,
                                                        const int16_t* __restrict__ Zin, const double* __restrict__ occ,
                                                        const double* __restrict__ Bf, int zmax, Geo* __restrict__ geo,
                                                        int set_geo, int* __restrict__ atom_bad, Atom32* __restrict__ a32,
                                                        AtomX* __restrict__ ax, float2* __restrict__ astep,
                                                        AtomR* __restrict__ ar, const float4* __restrict__ sctab)
{
    pdl_enter();
    __shared__ AtomShared sh;
    atoms_block(blockIdx.x, sh, atom_off, n_atoms, frac, Zin, occ, Bf, zmax, geo, set_geo, atom_bad, a32, ax, astep, ar,
                sctab);
}

// |g|^2 in the fixed order ((G11 hh + G22 kk) + G33 ll) + 2 ((G12 hk + G13 hl) + G23 kl).
__device__ __forceinline__ double q_exact(const double* gs, int h, int k, int l)
{
    const double hh = (double)(h * h), kk = (double)(k * k), ll = (double)(l * l);
    const double hk = (double)(h * k), hl = (double)(h * l), kl = (double)(k * l);
    const double diag = __dadd_rn(__dadd_rn(__dmul_rn(gs[0], hh), __dmul_rn(gs[1], kk)), __dmul_rn(gs[2], ll));
    const double off = __dadd_rn(__dadd_rn(__dmul_rn(gs[3], hk), __dmul_rn(gs[4], hl)), __dmul_rn(gs[5], kl));
    return __dadd_rn(diag, __dmul_rn(2.0, off));
}

// The l interval of column (h, k) that can hold |g|^2 <= r2max, computed in
// FP32 and widened by two on each side (a superset: every l in it is tested).
__device__ __forceinline__ void column_range(const float* gf, int L, int h, int k, float r2maxf, int& lo, int& hi)
{
    const float fh = (float)h, fk = (float)k;
    const float A = fmaf(gf[0] * fh, fh, fmaf(gf[1] * fk, fk, 2.f * gf[3] * fh * fk));
    const float b = fmaf(gf[4], fh, gf[5] * fk);
    const float R = r2maxf * 1.0001f;
    const float c = A - R;
    float disc = fmaf(b, b, -gf[2] * c);
    const float mag = fmaf(b, b, gf[2] * fabsf(c));
    lo = 1;
    hi = 0;
    if (disc < -1e-4f * mag) return;
    disc = fmaxf(disc, 0.f);
    const float sq = sqrtf(disc);
    const float inv = 1.f / gf[2];
    lo = (int)floorf((-b - sq) * inv) - 2;
    hi = (int)ceilf((-b + sq) * inv) + 2;
    if (lo < -L) lo = -L;
    if (hi > L) hi = L;
    if (h == 0 && k == 0 && lo < 1) lo = 1;  // half-space: (0, 0, l > 0)
}

__device__ __noinline__ int q_side_exact(const double* gs, int h, int k, int l, double r);

// Side of |g|^2 against a squared radius r for one (h, k, l): an FP32
// evaluation decides every candidate farther from r than a bound on its
// rounding error; the rest compare the fixed-order FP64 value (q_exact).
// Returns -1 (|g|^2 < r), 0 (equal) or 1 (|g|^2 > r).
__device__ __forceinline__ int q_side(const Geo& g, const double* gsg, int h, int k, int l, double r, float rf)
{
    const float* gf = g.gf;
    const float hh = (float)(h * h), kk = (float)(k * k), ll = (float)(l * l);
    const float hk = (float)(h * k), hl = (float)(h * l), kl = (float)(k * l);
    const float diag = fmaf(gf[2], ll, fmaf(gf[1], kk, gf[0] * hh));
    const float o1 = gf[3] * hk, o2 = gf[4] * hl, o3 = gf[5] * kl;
    const float qf = fmaf(2.f, o1 + o2 + o3, diag);
    const float qa = fmaf(2.f, fabsf(o1) + fabsf(o2) + fabsf(o3), diag);
    const float m = 4e-6f * qa + 1e-30f;
    if (qf > rf + m) return 1;
    if (qf < rf - m) return -1;
    return q_side_exact(gsg, h, k, l, r);
}

// The reflections of column (h, k) are the l of [a, b] outside [c, d] (c > d:
// the column misses the inner sphere). Along a column |g|^2 is a convex
// quadratic in l; its second difference 2 G*33 exceeds the rounding error of the
// fixed-order FP64 value by many orders of magnitude, so the l that pass the
// per-reflection test r2min <= |g|^2 <= r2max are exactly an interval minus an
// inner interval. Their ends are found by testing l inward from the FP32
// superset bounds of column_range, a few tests per column instead of one per l.
struct ColSpan {
    int a, b, c, d;
    __device__ int count() const { return a > b ? 0 : (b - a + 1) - (c <= d ? d - c + 1 : 0); }
    __device__ int first_part() const { return a > b ? 0 : (c <= d ? c - a : b - a + 1); }  // l in [a, c)
};

__device__ __forceinline__ ColSpan column_span(const Geo& g, const double* gsg, int h, int k, double r2min,
                                               double r2max, float r2minf, float r2maxf)
{
    ColSpan sp{1, 0, 1, 0};
    int lo, hi;
    column_range(g.gf, g.L, h, k, r2maxf, lo, hi);
    while (lo <= hi && q_side(g, gsg, h, k, lo, r2max, r2maxf) > 0) lo++;
    while (hi > lo && q_side(g, gsg, h, k, hi, r2max, r2maxf) > 0) hi--;
    if (lo > hi) return sp;
    sp.a = lo;
    sp.b = hi;
    if (r2min > 0.0) {
        int c0, d0;
        column_range(g.gf, g.L, h, k, r2minf, c0, d0);
        c0 = max(c0, lo);
        d0 = min(d0, hi);
        while (c0 <= d0 && q_side(g, gsg, h, k, c0, r2min, r2minf) >= 0) c0++;
        while (d0 > c0 && q_side(g, gsg, h, k, d0, r2min, r2minf) >= 0) d0--;
        if (c0 <= d0) {
            sp.c = c0;
            sp.d = d0;
        }
    }
    return sp;
}

// Columns of the half-space (h > 0, or h = 0 and k >= 0) in their emission
// order: h ascending, then k ascending; l ascending within a column.
__device__ __forceinline__ int n_columns(const Geo& g)
{
    return (g.status == XRD_OK && g.H >= 0) ? (g.K + 1) + g.H * (2 * g.K + 1) : 0;
}
__device__ __forceinline__ void column_hk(const Geo& g, int c, int& h, int& k)
{
    if (c <= g.K) {
        h = 0;
        k = c;
        return;
    }
    const int nk = 2 * g.K + 1, r = c - (g.K + 1);
    h = 1 + r / nk;
    k = r % nk - g.K;
}

// Runs: the structure-factor kernel gives each lane a run of at most kRunLen
// reflections that are consecutive in l within one column, so that it can step
// the phase factor exp(2 pi i g.x) from l to l + 1 by one complex rotation.
// Each of a column's (at most two) contiguous parts is cut into runs of kRunLen
// from its first l, the last one shorter. Run entries: (first reflection
// within the structure) << 3 | length.
constexpr int kRunLen = 4;
__device__ __forceinline__ int runs_of(int n) { return (n + kRunLen - 1) / kRunLen; }

// The exact comparison of a candidate within the FP32 error bound of a sphere
// surface, kept out of line so that the rare FP64 evaluation is a branch, not
// work that every caller does.
__device__ __noinline__ int q_side_exact(const double* gs, int h, int k, int l, double r)
{
    const double q = q_exact(gs, h, k, l);
    return q > r ? 1 : (q < r ? -1 : 0);
}

// Reflections and runs of column c.
__device__ __forceinline__ ColSpan column_counts(const Geo& g, const double* gsg, int c, double r2min, double r2max,
                                                 float r2minf, float r2maxf, bool runs, int& h, int& k, int& n,
                                                 int& nr)
{
    column_hk(g, c, h, k);
    const ColSpan sp = column_span(g, gsg, h, k, r2min, r2max, r2minf, r2maxf);
    n = sp.count();
    nr = 0;
    if (runs) {
        const int n1 = sp.first_part();
        nr = runs_of(n1) + runs_of(n - n1);
    }
    return sp;
}

__device__ __forceinline__ int warp_sum_int(int v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    return v;
}

// Work of the enumeration kernels: one warp per item. A structure of more than part_cols columns is split into
// parts of part_cols columns, which k_prep lists (GeomArgs::part_tab; Geo.pbase: the structure's first part) with
// room for part_cap parts; a structure that finds no room, or has fewer columns, is one item. A warp takes a part in
// about the time of part_cols / 32 steps of 32 columns, so a batch of few large cells, or one cell, fills the part.
// Measured with one warp or one CTA a structure before: the 50 A cell of 679 000 reflections 0.25 ms to count and
// 1.53 ms to emit, 256 cells of 15-40 A 0.13 and 1.37 ms; now 6 and 32 us, 17 and 106 us. 100 000 mixed cells in parts of
// 512 columns 0.21 and 0.72 ms, of 128 columns 0.19 and 0.55 ms; 5000 of them 45 and 153 us, and 20 and 64 us. Thin shells
// are where room runs out: 3000 cells of 20-30 A, 0.01 degrees of 2-theta, 12 000 reflections, 200 us a call with a warp a
// structure, 262 with room for a part a reflection, 173 with room for four; 2047 of them 177, 202 with narrow parts for some
// of them, 143 with wide ones for all.
// Items are claimed from a counter, the parts first: kClaimWide structures (or one part) at a time.
constexpr int kEnumMaxThreads = 1024;
constexpr int kClaimWide = 2;         // structures a claim takes in a batch of at least kClaimBatch, many for every warp
constexpr int kClaimBatch = 32768;    // (below, a warp with two structures that found no room is the last one to end)
constexpr int kWideBatch = 2048;      // enough structures to fill the GPU by themselves: parts of four chunks, which
constexpr int kPartColsWide = 128;    // bound the tail; below, every chunk of 32 columns is an item, since a warp's chunks
constexpr int kPartColsNarrow = 32;   // are a serial chain of about 5 us each
constexpr int kPartRoom = 64;         // unless there is room for fewer parts a structure: wide ones then, since a structure
                                      // that finds no room is one item, and the last one to end
static int enum_part_cols(int n_struct, int part_cap)
{
    return n_struct >= kWideBatch || part_cap < (int64_t)kPartRoom * n_struct ? kPartColsWide : kPartColsNarrow;
}

struct EnumItems {
    int nparts, n_struct, claim;
    int* ctr;
    // claims the next items: first is the first of n items (parts: 0 .. nparts - 1, then structures); n = 0 at the end
    __device__ __forceinline__ int next(int& n) const
    {
        const int lane = threadIdx.x & 31;
        int v = 0;
        if (lane == 0) v = atomicAdd(ctr, 1);
        v = __shfl_sync(0xffffffffu, v, 0);
        if (v < nparts) {
            n = 1;
            return v;
        }
        const int s0 = (v - nparts) * claim;
        n = max(0, min(claim, n_struct - s0));
        return nparts + s0;
    }
};

__device__ __forceinline__ EnumItems enum_items(int n_struct, const unsigned long long* part_ctr, int part_cap, int* ctr)
{
    return EnumItems{(int)min(*part_ctr, (unsigned long long)part_cap), n_struct, n_struct >= kClaimBatch ? kClaimWide : 1, ctr};
}

// The structure and the columns [c0, c1) of an item (none where bad says so); false where there is nothing to do (a structure that its
// parts cover, a slot of a structure that found no room)
__device__ __forceinline__ bool enum_item(const Geo* __restrict__ geo, const int2* __restrict__ part_tab, int nparts,
                                          int part_cols, int item, int& s, int& part, Geo& g, int& c0, int& c1,
                                          const int* __restrict__ bad = nullptr)
{
    part = -1;
    s = item - nparts;
    if (item < nparts) {
        const int2 t = part_tab[item];
        s = t.x;
        part = t.y;
        if (s < 0) return false;
    }
    g = geo[s];
    const int ncol = n_columns(g);
    c0 = 0;
    c1 = ncol;
    if (part >= 0) {
        c0 = part * part_cols;
        c1 = min(c0 + part_cols, ncol);
    } else if (g.pbase >= 0) {
        return false;
    }
    if (bad && bad[s]) c1 = c0;  // a structure with an invalid atom has no reflections
    return true;
}

// Record of a non-empty column of a chunk: its |g|^2 as a polynomial in l, q(l) = t + u l + G*33 l^2 with
// t = G*11 h^2 + G*22 k^2 + 2 G*12 hk and u = 2 G*13 h + 2 G*23 k in two-float arithmetic (about 1e-14 relative),
// and where its reflections and runs go.
struct __align__(16) ColRec {
    float th, tl, uh, ul;
    int a_off;      // first l minus the column's offset within the chunk
    int c, gap;     // first l of the inner gap (INT_MAX: none), its length
    uint32_t key0;  // the packed key of (h, k, 0)
    int off, roff;  // offset of the column's reflections and runs within the chunk
    int n, n1;      // its reflections, and those below the gap
};

__device__ __forceinline__ ColRec column_rec(const Geo& g, const ColSpan& sp, int h, int k, int n, int off, int roff)
{
    ColRec r;
    const F2 G11{g.gf[0], g.gl[0]}, G22{g.gf[1], g.gl[1]}, G12{2.f * g.gf[3], 2.f * g.gl[3]};
    const F2 G13{2.f * g.gf[4], 2.f * g.gl[4]}, G23{2.f * g.gf[5], 2.f * g.gl[5]};
    const F2 t = f2_add(f2_add(f2_mul_int(G11, (float)(h * h)), f2_mul_int(G22, (float)(k * k))),
                        f2_mul_int(G12, (float)(h * k)));
    const F2 u = f2_add(f2_mul_int(G13, (float)h), f2_mul_int(G23, (float)k));
    r.th = t.hi;
    r.tl = t.lo;
    r.uh = u.hi;
    r.ul = u.lo;
    r.a_off = sp.a - off;
    r.c = sp.c <= sp.d ? sp.c : INT_MAX;
    r.gap = sp.c <= sp.d ? sp.d - sp.c + 1 : 0;
    r.key0 = hkl_pack(h, k, 0);
    r.off = off;
    r.roff = roff;
    r.n = n;
    r.n1 = sp.first_part();
    return r;
}

// The item's entries of the structure-factor tile table from tile_off[s]: (s, first run) of each tile of 32 runs
// (runs), or (s, first reflection) of each tile of tile_refl reflections; entries t, t + nt, ...
__device__ __forceinline__ void write_tiles(int s, bool runs, int tile_refl, int64_t units, const int* __restrict__ tile_off,
                                            int2* __restrict__ tile_tab, int t, int nt)
{
    const int per = runs ? kRunsPerTile : tile_refl;
    const int ntl = (int)((units + per - 1) / per), t0 = tile_off[s];
    for (int i = t; i < ntl; i += nt) tile_tab[t0 + i] = make_int2(s, i * per);
}

// Writes |g|^2 and the packed (h, k, l) of every reflection of each structure
// (and its runs) from refl_off[s], and its tile-table entries. A warp takes an item's
// columns 32 at a time: each lane finds its column's span, a scan places the columns, the non-empty ones leave their
// records in shared memory, and the warp writes the chunk's reflections as one flat, coalesced range. Which column
// owns position p0 + lane comes from one bit per column start in [p0, p0 + 32), gathered by a warp-wide OR: the
// owner is the number of starts at or below the position (a bisection over 32 offsets cost five dependent
// shared-memory loads per reflection). A reflection that starts a run writes the run's entry. The
// output order is the column order above, l ascending, whatever the launch shape.
template <bool RUNS>
__global__ void __launch_bounds__(kEnumMaxThreads) k_emit(const Geo* __restrict__ geo, int n_struct, double r2min,
                                                          double r2max, float r2minf, float r2maxf,
                                                          int tile_refl, const int64_t* __restrict__ refl_off,
                                                          const int64_t* __restrict__ run_cnt,
                                                          const int* __restrict__ abort_flag, double* __restrict__ q,
                                                          uint32_t* __restrict__ key, int* __restrict__ runs,
                                                          const int* __restrict__ tile_off, int2* __restrict__ tile_tab,
                                                          int* __restrict__ ctr, const unsigned long long* __restrict__ part_ctr,
                                                          const int2* __restrict__ part_tab,
                                                          const int2* __restrict__ part_cnt, int part_cap, int part_cols)
{
    pdl_enter();
    extern __shared__ __align__(16) unsigned char esm[];
    if (*abort_flag) return;
    const int lane = threadIdx.x & 31;
    ColRec* const rec = (ColRec*)esm + 32 * (threadIdx.x >> 5);
    const unsigned le = 0xffffffffu >> (31 - lane);
    const EnumItems items = enum_items(n_struct, part_ctr, part_cap, ctr);
    for (;;) {
        int nit;
        const int first = items.next(nit);
        if (nit == 0) break;
        for (int it = first; it < first + nit; it++) {
            int s, part, c_lo, c_hi;
            Geo g;
            if (!enum_item(geo, part_tab, items.nparts, part_cols, it, s, part, g, c_lo, c_hi)) continue;
            const int64_t base = refl_off[s], cap = refl_off[s + 1] - base;
            int done = 0, done_runs = 0;  // the structure's reflections and runs before this chunk
            {
                const int np = part < 0 ? 1 : (n_columns(g) + part_cols - 1) / part_cols;
                if (tile_tab)
                    write_tiles(s, RUNS, tile_refl, RUNS ? run_cnt[s] : cap, tile_off, tile_tab,
                                32 * max(part, 0) + lane, 32 * np);
                if (part > 0) {
                    for (int i = lane; i < part; i += 32) {
                        const int2 v = part_cnt[g.pbase + i];
                        done += v.x;
                        done_runs += v.y;
                    }
                    done = warp_sum_int(done);
                    if (RUNS) done_runs = warp_sum_int(done_runs);
                }
            }
            if (cap <= 0) continue;
            const F2 g33{g.gf[2], g.gl[2]};
            for (int c0 = c_lo; c0 < c_hi; c0 += 32) {
                const int c = c0 + lane;
                int h = 0, k = 0, n = 0, nr = 0;
                ColSpan sp{1, 0, 1, 0};
                if (c < c_hi)
                    sp = column_counts(g, geo[s].gs, c, r2min, r2max, r2minf, r2maxf, RUNS, h, k, n, nr);
                const int im = warp_incl_scan(n), imr = RUNS ? warp_incl_scan(nr) : 0;
                const int off = im - n;
                const unsigned full = __ballot_sync(0xffffffffu, n > 0);
                if (n > 0) rec[__popc(full & le) - 1] = column_rec(g, sp, h, k, n, off, imr - nr);
                const int tot = __shfl_sync(0xffffffffu, im, 31);
                __syncwarp();
                int started = 0;  // non-empty columns that start before p0
                for (int p0 = 0; p0 < tot; p0 += 32) {
                    const int d = off - p0;
                    const unsigned starts = __reduce_or_sync(0xffffffffu, (n > 0 && d >= 0 && d < 32) ? 1u << d : 0u);
                    const ColRec r = rec[max(started + __popc(starts & le) - 1, 0)];
                    started += __popc(starts);
                    const int p = p0 + lane;
                    if (p >= tot) continue;
                    int l = r.a_off + p;
                    if (l >= r.c) l += r.gap;
                    const int64_t pos = done + p;
                    if (pos < cap) {
                        const float fl = (float)l;
                        const F2 v = f2_add(f2_add(F2{r.th, r.tl}, f2_mul_int(g33, fl * fl)),
                                            f2_mul_int(F2{r.uh, r.ul}, fl));
                        q[base + pos] = f2d_fast(v.hi) + f2d_fast(v.lo);
                        key[base + pos] = r.key0 + l;
                    }
                    if (RUNS) {
                        const bool above = p - r.off >= r.n1;  // past the inner gap
                        const int j = p - r.off - (above ? r.n1 : 0), nn = above ? r.n - r.n1 : r.n1;
                        if ((j & (kRunLen - 1)) == 0) {
                            const int64_t rpos = done_runs + r.roff + (above ? runs_of(r.n1) : 0) + j / kRunLen;
                            if (rpos < cap) runs[base + rpos] = ((done + p) << 3) | min(kRunLen, nn - j);
                        }
                    }
                }
                done += tot;
                if (RUNS) done_runs += __shfl_sync(0xffffffffu, imr, 31);
                __syncwarp();  // the records are read before the next chunk rewrites them
            }
        }
    }
}

// Single block. Every pass walks the batch in chunks of kScanItems * blockDim
// structures (or positions in the largest-first order): coalesced loads into
// registers, a transpose through shared memory when a pass needs a prefix,
// and warp-aggregated shared-memory atomics where it needs ranks.
//  1. reflection offsets (64-bit exclusive scan of the counts), the capacity
//     check and the per-structure status;
//  2. in the largest-first order (k_order), each structure's first tile and
//     the post-processing size-class lists (post_class; within a class the
//     order follows the chunks).
// The tile table itself is written by k_emit, each item its share of its structure's entries.
constexpr int kOrderBins = 4096;
constexpr int kScanThreads = 1024;
constexpr int kScanItems = 4;

template <int BINS = kOrderBins>
__device__ __forceinline__ int order_bin(const int64_t* __restrict__ atom_off, int s)
{
    const long long na = atom_off[s + 1] - atom_off[s];
    return BINS - 1 - (int)min(max(na, 0LL), (long long)(BINS - 1));
}

// Rank of this lane among the lanes of its warp with the same key, and the
// base the group's leader obtained with one shared-memory atomicAdd on ctr[key].
__device__ __forceinline__ int warp_aggregated_slot(int* ctr, int key, bool active)
{
    const unsigned act = __ballot_sync(0xffffffffu, active);
    if (!active) return 0;
    const unsigned peers = __match_any_sync(act, key);
    const int lane = threadIdx.x & 31;
    const int leader = __ffs(peers) - 1;
    int base = 0;
    if (lane == leader) base = atomicAdd(&ctr[key], __popc(peers));
    base = __shfl_sync(peers, base, leader);
    return base + __popc(peers & ((1u << lane) - 1u));
}

// Bins of the order by reflection count, largest first: a quarter octave each, the last for none.
constexpr int kCountBins = 128;
__device__ __forceinline__ int count_bin(long long r)
{
    return r <= 0 ? kCountBins - 1 : max(kCountBins - 2 - (int)(4.f * log2f((float)r)), 0);
}

struct ScanArgs {
    const int64_t* run_cnt;
    int tile_refl;
    int64_t cap_refl;
    int64_t* refl_off;
    int* tile_off;
    const int* order;
    int* cls_list;
    int* abort_flag;
    int64_t* totals;
    int32_t* status;
    unsigned long long* work;
    int* aorder;     // [n] the structures by reflection count, largest first (or nullptr); within a bin the order is
                     // arbitrary: nothing but the load balance depends on it
    const int* bad;  // structures with an invalid atom become invalid here (or nullptr)
    unsigned long long* sums;  // not nullptr: no scan, but the counts' sum, largest, and tiles of tile_refl and of half as
                               // many reflections into sums[0..3]
};
struct ScanShared {
    long long ws[33];
    int ccnt[kPostClasses];
    int bins[kCountBins];
};

// Exclusive scan of the kCountBins bins by the first warp
__device__ __forceinline__ void scan_count_bins(int* bins)
{
    if (threadIdx.x >= 32) return;
    constexpr int per = kCountBins / 32;
    int v[per], sum = 0;
#pragma unroll
    for (int j = 0; j < per; j++) sum += v[j] = bins[per * threadIdx.x + j];
    int run = warp_incl_scan(sum) - sum;
#pragma unroll
    for (int j = 0; j < per; j++) {
        bins[per * threadIdx.x + j] = run;
        run += v[j];
    }
}

// buf: kScanItems * blockDim long longs of shared memory. The counts are read past the L1 cache: the CTA that runs
// this may be one of the kernel that wrote them.
// ORDER: also the order by reflection count, if sa.aorder.
template <bool ORDER>
__device__ __forceinline__ void scan_refl_block(const int64_t* cnt, Geo* __restrict__ geo, int n,
                                                const ScanArgs& sa, ScanShared& sh, long long* buf)
{
    const int64_t* const run_cnt = sa.run_cnt;
    const int tile_refl = sa.tile_refl;
    const int64_t cap_refl = sa.cap_refl;
    int64_t* const refl_off = sa.refl_off;
    int* const tile_off = sa.tile_off;
    const int* const order = sa.order;
    int* const cls_list = sa.cls_list;
    int* const abort_flag = sa.abort_flag;
    int64_t* const totals = sa.totals;
    int32_t* const status = sa.status;
    unsigned long long* const work = sa.work;
    long long* const ws = sh.ws;
    int* const ccnt = sh.ccnt;
    const int nt = blockDim.x, tid = threadIdx.x, CH = kScanItems * nt;
    int* const aorder = ORDER ? sa.aorder : nullptr;
    int* const bins = sh.bins;
    long long tot;
    if (aorder) {
        for (int b = tid; b < kCountBins; b += nt) bins[b] = 0;
        __syncthreads();
    }
    // 1. reflection offsets in structure order, the status of each structure, and how many have how many reflections
    long long carry = 0, bad = 0;
    for (int base = 0; base < n; base += CH) {
        long long v[kScanItems];
        int st[kScanItems];
#pragma unroll
        for (int u = 0; u < kScanItems; u++) {
            const int i = base + u * nt + tid;
            v[u] = i < n ? __ldcg((const long long*)cnt + i) : 0;
            st[u] = i < n ? geo[i].status : XRD_OK;
            if (i < n && sa.bad && sa.bad[i]) {
                st[u] = XRD_EINVAL;
                geo[i].status = XRD_EINVAL;
            }
            if (aorder && i < n) atomicAdd(&bins[count_bin(v[u])], 1);
        }
        chunk_scan<kScanItems>(v, buf, ws, &tot);
#pragma unroll
        for (int u = 0; u < kScanItems; u++) {
            const int i = base + u * nt + tid;
            if (i < n) {
                refl_off[i] = carry + v[u];
                status[i] = st[u];
            }
            bad += st[u] != XRD_OK;
        }
        carry += tot;
    }
    const long long total = carry;
    const bool over = total > cap_refl;
    block_prefix_ll(bad, ws, &tot);
    const long long nbad = over ? n : tot;
    if (over)
        for (int i = tid; i < n; i += nt) status[i] = XRD_ECAPACITY;
    if (tid < kPostClasses) ccnt[tid] = 0;
    if (aorder) scan_count_bins(bins);
    __syncthreads();
    // 2. tiles and size classes in the largest-first order
    long long tcarry = 0;
    for (int base = 0; base < n; base += CH) {
        long long v[kScanItems];
        int sv[kScanItems];
#pragma unroll
        for (int u = 0; u < kScanItems; u++) {
            const int p = base + u * nt + tid;
            sv[u] = p < n ? order[p] : -1;
        }
        long long c[kScanItems];
#pragma unroll
        for (int u = 0; u < kScanItems; u++) {
            c[u] = sv[u] >= 0 ? __ldcg((const long long*)cnt + sv[u]) : 0;
            // tiles of 32 runs, or of tile_refl reflections
            v[u] = sv[u] < 0 ? 0 : (tile_refl > 0 ? (c[u] + tile_refl - 1) / tile_refl
                                                  : (__ldcg((const long long*)run_cnt + sv[u]) + kRunsPerTile - 1) / kRunsPerTile);
        }
        chunk_scan<kScanItems>(v, buf, ws, &tot);
#pragma unroll
        for (int u = 0; u < kScanItems; u++) {
            const int p = base + u * nt + tid;
            if (p < n) tile_off[sv[u]] = (int)(tcarry + v[u]);  // first tile of the structure
            if (aorder && p < n) aorder[atomicAdd(&bins[count_bin(c[u])], 1)] = sv[u];
            if (!over && cls_list) {
                const int k = post_class(c[u]);
                const int slot = warp_aggregated_slot(ccnt, k, p < n);
                if (p < n) cls_list[(int64_t)k * n + slot] = sv[u];
            }
        }
        tcarry += tot;
        __syncthreads();  // this chunk's class slots are taken before the next chunk's
    }
    if (tid == 0) {
        if (work) {  // for xrd_work_counts: the tiles and the tile mode of this call
            work[0] = (unsigned long long)tcarry;
            work[1] = tile_refl > 0 ? 0ull : 1ull;
        }
        refl_off[n] = total;
        tile_off[n] = over ? 0 : (int)tcarry;
        for (int k = 0; k < kPostClasses; k++) abort_flag[kFlagClsCnt + k] = over ? 0 : ccnt[k];
        totals[0] = total;
        totals[1] = 0;
        totals[2] = 0;
        totals[3] = nbad;
        *abort_flag = over;
    }
}

__global__ void __launch_bounds__(kScanThreads) k_scan_refl(const int64_t* __restrict__ cnt, Geo* __restrict__ geo,
                                                            int n, const ScanArgs sa)
{
    pdl_enter();
    __shared__ ScanShared sh;
    __shared__ __align__(16) long long buf[kScanItems * kScanThreads];
    scan_refl_block<true>(cnt, geo, n, sa, sh, buf);
}

// Reflection (and, with RUNS, run) counts per structure, and of every part (k_prep has zeroed the counts of a
// structure in parts). ctr: zero at launch. done: CTAs finished (zero at launch), or null: no scan.
template <bool RUNS>
__global__ void __launch_bounds__(kEnumMaxThreads) k_count(Geo* geo, int n_struct, double r2min,
                                                           double r2max, float r2minf, float r2maxf,
                                                           int64_t* __restrict__ cnt, int64_t* __restrict__ run_cnt,
                                                           int* __restrict__ ctr, const unsigned long long* __restrict__ part_ctr,
                                                           const int2* __restrict__ part_tab,
                                                           int2* __restrict__ part_cnt, int part_cap, int part_cols,
                                                           const ScanArgs scan, int* __restrict__ done,
                                                           const int* __restrict__ bad)
{
    pdl_enter();
    const int lane = threadIdx.x & 31;
    const EnumItems items = enum_items(n_struct, part_ctr, part_cap, ctr);
    for (;;) {
        int m;
        const int first = items.next(m);
        if (m == 0) break;
        for (int it = first; it < first + m; it++) {
            int s, part, c0, c1;
            Geo g;
            if (!enum_item(geo, part_tab, items.nparts, part_cols, it, s, part, g, c0, c1, bad)) continue;
            int local = 0, local_runs = 0;
            for (int c = c0 + lane; c < c1; c += 32) {
                int h, k, n, nr;
                column_counts(g, geo[s].gs, c, r2min, r2max, r2minf, r2maxf, RUNS, h, k, n, nr);
                local += n;
                local_runs += nr;
            }
            local = warp_sum_int(local);
            if (RUNS) local_runs = warp_sum_int(local_runs);
            if (lane != 0) continue;
            if (part < 0) {
                cnt[s] = local;
                if (RUNS && run_cnt) run_cnt[s] = local_runs;
            } else {
                part_cnt[it] = make_int2(local, local_runs);
                atomicAdd((unsigned long long*)(cnt + s), (unsigned long long)local);
                if (RUNS && run_cnt) atomicAdd((unsigned long long*)(run_cnt + s), (unsigned long long)local_runs);
            }
        }
    }
    if (!done) return;
    // the CTA that finishes last scans the counts (a launch less in a small batch's chain), or adds them up
    extern __shared__ __align__(16) long long scan_buf[];
    __shared__ ScanShared sh;
    __shared__ int last;
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) last = atomicAdd(done, 1) == (int)gridDim.x - 1;
    __syncthreads();
    if (!last) return;
    __threadfence();
    if (scan.sums) {
        long long sum = 0, most = 0, tiles = 0, half = 0, t;
        for (int i = threadIdx.x; i < n_struct; i += blockDim.x) {
            const long long c = __ldcg((const long long*)cnt + i);
            sum += c;
            most = max(most, c);
            tiles += (c + scan.tile_refl - 1) / scan.tile_refl;
            half += (2 * c + scan.tile_refl - 1) / scan.tile_refl;
        }
        block_prefix_ll(sum, sh.ws, &t);
        if (threadIdx.x == 0) scan.sums[0] = t;
        block_prefix_ll(tiles, sh.ws, &t);
        if (threadIdx.x == 0) scan.sums[2] = t;
        block_prefix_ll(half, sh.ws, &t);
        if (threadIdx.x == 0) scan.sums[3] = t;
        const unsigned long long m = block_max_u64(most, (unsigned long long*)sh.ws);
        if (threadIdx.x == 0) scan.sums[1] = m;
        return;
    }
    scan_refl_block<false>(cnt, geo, n_struct, scan, sh, scan_buf);
}

// Multi-block form of k_scan_refl for batches of more than two chunks (one
// chunk of kScanItems * kScanThreads structures per CTA): k_scan_refl_parts
// writes each chunk's sums (reflections, invalid structures, tiles in the
// largest-first order, structures per size class); k_scan_refl_final offsets
// every chunk by the sums of the chunks before it and repeats the single-block
// passes on its own chunk. Class-list slots follow the chunk order.
constexpr int kScanPartWords = 3 + kPostClasses;  // refl, bad, tiles, class counts

__device__ __forceinline__ long long tiles_of(const int64_t* __restrict__ run_cnt, int s, long long c, int tile_refl)
{
    return tile_refl > 0 ? (c + tile_refl - 1) / tile_refl : (run_cnt[s] + kRunsPerTile - 1) / kRunsPerTile;
}

__global__ void __launch_bounds__(kScanThreads) k_scan_refl_parts(const int64_t* __restrict__ cnt,
                                                                  const int64_t* __restrict__ run_cnt,
                                                                  const Geo* __restrict__ geo, int n, int tile_refl,
                                                                  const int* __restrict__ order,
                                                                  long long* __restrict__ parts,
                                                                  int* __restrict__ oparts)
{
    pdl_enter();
    __shared__ long long ws[33];
    __shared__ int cc[kPostClasses], bins[kCountBins];
    const int nt = blockDim.x, tid = threadIdx.x, base = blockIdx.x * kScanItems * nt;
    if (tid < kPostClasses) cc[tid] = 0;
    if (tid < kCountBins) bins[tid] = 0;
    __syncthreads();
    long long refl = 0, bad = 0, tiles = 0;
#pragma unroll
    for (int u = 0; u < kScanItems; u++) {
        const int i = base + u * nt + tid;
        if (i < n) {
            refl += cnt[i];
            bad += geo[i].status != XRD_OK;
            const int sv = order[i];  // position i of the largest-first order
            const long long c = cnt[sv];
            tiles += tiles_of(run_cnt, sv, c, tile_refl);
            atomicAdd(&cc[post_class(c)], 1);
            if (oparts) atomicAdd(&bins[count_bin(c)], 1);
        }
    }
    long long t;
    block_prefix_ll(refl, ws, &t);
    refl = t;
    block_prefix_ll(bad, ws, &t);
    bad = t;
    block_prefix_ll(tiles, ws, &t);
    tiles = t;
    if (oparts && tid < kCountBins) oparts[(int64_t)blockIdx.x * kOrderBins + tid] = bins[tid];
    if (tid == 0) {
        long long* o = parts + (int64_t)blockIdx.x * kScanPartWords;
        o[0] = refl;
        o[1] = bad;
        o[2] = tiles;
        for (int k = 0; k < kPostClasses; k++) o[3 + k] = cc[k];
    }
}

__global__ void __launch_bounds__(kScanThreads) k_scan_refl_final(const int64_t* __restrict__ cnt,
                                                                  const int64_t* __restrict__ run_cnt,
                                                                  const Geo* __restrict__ geo, int n, int tile_refl,
                                                                  int64_t cap_refl, int64_t* __restrict__ refl_off,
                                                                  int* __restrict__ tile_off, const int* __restrict__ order,
                                                                  int* __restrict__ cls_list, int* __restrict__ abort_flag,
                                                                  int64_t* __restrict__ totals, int32_t* __restrict__ status,
                                                                  unsigned long long* __restrict__ work,
                                                                  const long long* __restrict__ parts,
                                                                  const int* __restrict__ oparts, int* __restrict__ aorder)
{
    pdl_enter();
    __shared__ long long ws[33];
    __shared__ __align__(16) long long buf[kScanItems * kScanThreads];
    __shared__ long long pre[kScanPartWords], all[kScanPartWords];
    __shared__ int ccnt[kPostClasses], bins[kCountBins];
    const int nt = blockDim.x, tid = threadIdx.x, b = blockIdx.x, base = b * kScanItems * nt;
    const int nch = gridDim.x;
    if (tid < kScanPartWords) {  // sums of the chunks before this one, and of all chunks
        long long p = 0, a = 0;
        for (int c = 0; c < nch; c++) {
            const long long v = parts[(int64_t)c * kScanPartWords + tid];
            p += c < b ? v : 0;
            a += v;
        }
        pre[tid] = p;
        all[tid] = a;
    }
    if (tid < kPostClasses) ccnt[tid] = 0;
    int before = 0;  // structures of this thread's bin in the chunks before this one
    if (aorder && tid < kCountBins) {
        int a = 0;
        for (int c = 0; c < nch; c++) {
            const int v = oparts[(int64_t)c * kOrderBins + tid];
            before += c < b ? v : 0;
            a += v;
        }
        bins[tid] = a;
    }
    __syncthreads();
    if (aorder) {
        scan_count_bins(bins);
        __syncthreads();
        if (tid < kCountBins) bins[tid] += before;  // read after the scans below
    }
    const long long total = all[0];
    const bool over = total > cap_refl;
    long long v[kScanItems], tot;
    int st[kScanItems];
    // 1. reflection offsets and status
#pragma unroll
    for (int u = 0; u < kScanItems; u++) {
        const int i = base + u * nt + tid;
        v[u] = i < n ? cnt[i] : 0;
        st[u] = i < n ? geo[i].status : XRD_OK;
    }
    chunk_scan<kScanItems>(v, buf, ws, &tot);
#pragma unroll
    for (int u = 0; u < kScanItems; u++) {
        const int i = base + u * nt + tid;
        if (i < n) {
            refl_off[i] = pre[0] + v[u];
            status[i] = over ? XRD_ECAPACITY : st[u];
        }
    }
    // 2. first tile of each structure and the size-class lists, in the largest-first order
    int sv[kScanItems];
    long long c[kScanItems];
#pragma unroll
    for (int u = 0; u < kScanItems; u++) {
        const int p = base + u * nt + tid;
        sv[u] = p < n ? order[p] : -1;
        c[u] = sv[u] >= 0 ? cnt[sv[u]] : 0;
        v[u] = sv[u] < 0 ? 0 : tiles_of(run_cnt, sv[u], c[u], tile_refl);
    }
    chunk_scan<kScanItems>(v, buf, ws, &tot);
#pragma unroll
    for (int u = 0; u < kScanItems; u++) {
        const int p = base + u * nt + tid;
        if (p < n) tile_off[sv[u]] = (int)(pre[2] + v[u]);
        if (aorder && p < n) aorder[atomicAdd(&bins[count_bin(c[u])], 1)] = sv[u];
        if (!over && cls_list) {
            const int k = post_class(c[u]);
            const int slot = warp_aggregated_slot(ccnt, k, p < n);
            if (p < n) cls_list[(int64_t)k * n + (int)pre[3 + k] + slot] = sv[u];
        }
    }
    if (b == 0 && tid == 0) {
        if (work) {
            work[0] = (unsigned long long)all[2];
            work[1] = tile_refl > 0 ? 0ull : 1ull;
        }
        refl_off[n] = total;
        tile_off[n] = over ? 0 : (int)all[2];
        for (int k = 0; k < kPostClasses; k++) abort_flag[kFlagClsCnt + k] = over ? 0 : (int)all[3 + k];
        totals[0] = total;
        totals[1] = 0;
        totals[2] = 0;
        totals[3] = over ? n : all[1];
        *abort_flag = over;
    }
}

// Largest-first order of the structures: a counting sort on the atom count
// (which sets the cost of a structure-factor tile), in descending order; one
// block, warp-aggregated shared-memory atomics, so structures of one bin keep
// the order of their warp. It depends on the input only and runs beside the
// enumeration.
template <int BINS>
__device__ __forceinline__ void order_block(const int64_t* __restrict__ atom_off, int n, int* __restrict__ order,
                                            int* bins, int* tmp)
{
    const int nt = blockDim.x, tid = threadIdx.x, CH = kScanItems * nt;
    for (int b = tid; b < BINS; b += nt) bins[b] = 0;
    __syncthreads();
    for (int base = 0; base < n; base += CH) {
        int b[kScanItems];
#pragma unroll
        for (int u = 0; u < kScanItems; u++) {
            const int i = base + u * nt + tid;
            b[u] = i < n ? order_bin<BINS>(atom_off, i) : 0;
        }
#pragma unroll
        for (int u = 0; u < kScanItems; u++) warp_aggregated_slot(bins, b[u], base + u * nt + tid < n);
    }
    __syncthreads();
    block_excl_scan(bins, BINS, tmp);
    for (int base = 0; base < n; base += CH) {
        int b[kScanItems];
#pragma unroll
        for (int u = 0; u < kScanItems; u++) {
            const int i = base + u * nt + tid;
            b[u] = i < n ? order_bin<BINS>(atom_off, i) : 0;
        }
#pragma unroll
        for (int u = 0; u < kScanItems; u++) {
            const int i = base + u * nt + tid;
            const int slot = warp_aggregated_slot(bins, b[u], i < n);
            if (i < n) order[slot] = i;
        }
    }
}

__global__ void __launch_bounds__(kScanThreads) k_order(const int64_t* __restrict__ atom_off, int n,
                                                        int* __restrict__ order)
{
    pdl_enter();
    __shared__ int bins[kOrderBins];
    __shared__ int tmp[66];
    order_block<kOrderBins>(atom_off, n, order, bins, tmp);
}

// The whole input-only front of a small batch in one launch: block 0 forms the largest-first order, block 1 the
// coefficients, the next blocks the cells (16 structures each), the others pack the atoms of one structure each. One launch
// instead of four on two streams: a small batch is bound by its chain of launches. Taken up to kFrontMax structures of
// kFrontAtoms atoms on average; beyond, packing the atoms takes longer than counting the reflections, and the two
// run side by side on two streams instead.
constexpr int kFrontBins = 512;  // atom counts above this share a bin: the order only balances the load
struct FrontArgs {
    GeomArgs g;
    EnumParts ep;
    int prep_blocks;
};
__global__ void __launch_bounds__(kAtomThreads) k_front(const FrontArgs f)
{
    pdl_enter();
    __shared__ union {
        AtomShared at;
        struct {
            int bins[kFrontBins], tmp[66];
        } ord;
    } sh;
    const GeomArgs& g = f.g;
    const int b = blockIdx.x;
    if (b == 0) {
        order_block<kFrontBins>(g.atom_off, g.n_struct, g.order, sh.ord.bins, sh.ord.tmp);
    } else if (b == 1) {
        coef_block(g.coef, g.zmax, g.coef32, g.cdd);
    } else if (b <= 1 + f.prep_blocks) {
        prep_thread<8>((b - 2) * kAtomThreads + threadIdx.x, g.lattice, g.n_struct, g.rmax, g.geo, g.imax, g.out_flags,
                       f.ep);
    } else {
        atoms_block(b - 2 - f.prep_blocks, sh.at, g.atom_off, g.n_atoms, g.frac, g.Z, g.occ, g.B, g.zmax, g.geo, 0,
                    g.atom_bad, g.atom32, g.atomx, g.runs_mode ? g.astep : nullptr, g.atomr, g.sctab);
    }
}

// Multi-block form of the same order (more than two chunks of kScanItems *
// kScanThreads structures). k_order_parts histograms each chunk into
// oparts[chunk][bin]; k_order_final starts each bin of a chunk after all
// structures of the earlier bins and those of the same bin in earlier chunks,
// then scatters the chunk as k_order does.
__global__ void __launch_bounds__(kScanThreads) k_order_parts(const int64_t* __restrict__ atom_off, int n,
                                                              int* __restrict__ oparts)
{
    pdl_enter();
    __shared__ int bins[kOrderBins];
    const int nt = blockDim.x, tid = threadIdx.x, base = blockIdx.x * kScanItems * nt;
    for (int b = tid; b < kOrderBins; b += nt) bins[b] = 0;
    __syncthreads();
    int b[kScanItems];
#pragma unroll
    for (int u = 0; u < kScanItems; u++) {
        const int i = base + u * nt + tid;
        b[u] = i < n ? order_bin(atom_off, i) : 0;
    }
#pragma unroll
    for (int u = 0; u < kScanItems; u++) warp_aggregated_slot(bins, b[u], base + u * nt + tid < n);
    __syncthreads();
    for (int j = tid; j < kOrderBins; j += nt) oparts[(size_t)blockIdx.x * kOrderBins + j] = bins[j];
}

__global__ void __launch_bounds__(kScanThreads) k_order_final(const int64_t* __restrict__ atom_off, int n,
                                                              const int* __restrict__ oparts, int* __restrict__ order)
{
    pdl_enter();
    __shared__ int bins[kOrderBins], before[kOrderBins];
    __shared__ int tmp[66];
    const int nt = blockDim.x, tid = threadIdx.x, ch = blockIdx.x, nch = gridDim.x, base = ch * kScanItems * nt;
    for (int j = tid; j < kOrderBins; j += nt) {
        int tot = 0, bef = 0;
        for (int c = 0; c < nch; c++) {
            const int v = oparts[(size_t)c * kOrderBins + j];
            tot += v;
            bef += c < ch ? v : 0;
        }
        bins[j] = tot;
        before[j] = bef;
    }
    __syncthreads();
    block_excl_scan(bins, kOrderBins, tmp);
    for (int j = tid; j < kOrderBins; j += nt) bins[j] += before[j];
    __syncthreads();
    int b[kScanItems];
#pragma unroll
    for (int u = 0; u < kScanItems; u++) {
        const int i = base + u * nt + tid;
        b[u] = i < n ? order_bin(atom_off, i) : 0;
    }
#pragma unroll
    for (int u = 0; u < kScanItems; u++) {
        const int i = base + u * nt + tid;
        const int slot = warp_aggregated_slot(bins, b[u], i < n);
        if (i < n) order[slot] = i;
    }
}

template <typename... P, typename... A>
static void launch_k(bool pdl, void (*k)(P...), dim3 grid, dim3 block, cudaStream_t st, A... args)
{
    if (pdl) launch_pdl(k, grid, block, 0, st, args...);
    else k<<<grid, block, 0, st>>>(static_cast<P>(args)...);
}

static EnumParts enum_parts(const GeomArgs& a)
{
    return EnumParts{(unsigned long long*)(a.enum_ctr + kPartCtr), enum_part_cols(a.n_struct, a.part_cap), a.part_cap, a.part_tab, a.refl_cnt, a.run_cnt};
}

static void prep_launch(bool pdl, const GeomArgs& a, cudaStream_t st)
{
    const int n = a.n_struct;
    if (n <= kPrepWideMax)  // 4 structures per CTA
        launch_k(pdl, k_prep<8>, (n + 3) / 4, 32, st, a.lattice, n, a.rmax, a.geo, a.imax, a.out_flags, enum_parts(a));
    else
        launch_k(pdl, k_prep<1>, (n + 127) / 128, 128, st, a.lattice, n, a.rmax, a.geo, a.imax, a.out_flags,
                 enum_parts(a));
}

// Structure-factor work of the last call (for xrd_work_counts): terms = sum of
// reflections x atoms; phase seeds = the same with strided tiles, runs x atoms
// with runs; out[0..2] = terms, seeds, tiles (out zeroed by the caller).
__global__ void __launch_bounds__(256) k_work(const int64_t* __restrict__ cnt, const int64_t* __restrict__ run_cnt,
                                              const int64_t* __restrict__ atom_off, int n,
                                              const unsigned long long* __restrict__ work,
                                              unsigned long long* __restrict__ out)
{
    __shared__ unsigned long long red[2][8];
    const bool runs = work[1] != 0;
    unsigned long long t = 0, sd = 0;
    for (int s = blockIdx.x * blockDim.x + threadIdx.x; s < n; s += gridDim.x * blockDim.x) {
        const unsigned long long na = (unsigned long long)(atom_off[s + 1] - atom_off[s]);
        t += (unsigned long long)cnt[s] * na;
        sd += (unsigned long long)(runs ? run_cnt[s] : cnt[s]) * na;
    }
    for (int o = 16; o > 0; o >>= 1) {
        t += __shfl_xor_sync(0xffffffffu, t, o);
        sd += __shfl_xor_sync(0xffffffffu, sd, o);
    }
    const int w = threadIdx.x >> 5;
    if ((threadIdx.x & 31) == 0) {
        red[0][w] = t;
        red[1][w] = sd;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int i = 1; i < (int)(blockDim.x >> 5); i++) {
            t += red[0][i];
            sd += red[1][i];
        }
        atomicAdd(&out[0], t);
        atomicAdd(&out[1], sd);
        if (blockIdx.x == 0) out[2] = work[0];
    }
}

void launch_work(const GeomArgs& a, unsigned long long* out, cudaStream_t st)
{
    if (a.n_struct > 0)
        k_work<<<min((a.n_struct + 255) / 256, 1024), 256, 0, st>>>(a.refl_cnt, a.run_cnt, a.atom_off, a.n_struct,
                                                                   a.work, out);
}

constexpr int kFrontMax = 2048, kFrontAtoms = 128;
bool front_fused(int n_struct, int64_t n_atoms) { return n_struct <= kFrontMax && n_atoms <= (int64_t)n_struct * kFrontAtoms; }

void launch_front(const GeomArgs& a, cudaStream_t st)
{
    if (a.n_struct <= 0) return;
    FrontArgs f{a, enum_parts(a), (8 * a.n_struct + kAtomThreads - 1) / kAtomThreads};
    k_front<<<2 + f.prep_blocks + a.n_struct, kAtomThreads, 0, st>>>(f);
}

void launch_prep(const GeomArgs& a, cudaStream_t st, bool pdl)
{
    if (a.n_struct > 0) prep_launch(pdl, a, st);
}

void launch_coef(const GeomArgs& a, cudaStream_t st, bool pdl)
{
    launch_k(pdl, k_coef, 1, 256, st, a.coef, a.zmax, a.coef32, a.cdd);
}

void launch_atoms(const GeomArgs& a, cudaStream_t st, bool pdl)
{
    if (a.n_struct > 0)
        launch_k(pdl, k_atoms, a.n_struct, kAtomThreads, st, a.atom_off, a.n_atoms, a.frac, a.Z, a.occ, a.B, a.zmax, a.geo,
                 a.atoms_set_geo, a.atom_bad, a.atom32, a.atomx, a.runs_mode ? a.astep : (float2*)nullptr, a.atomr,
                 a.sctab);
}

void launch_order(const GeomArgs& a, cudaStream_t st, bool pdl)
{
    if (a.n_struct <= 0) return;
    const int nch = (a.n_struct + kScanItems * kScanThreads - 1) / (kScanItems * kScanThreads);
    if (nch <= 2 || !a.oparts) {
        launch_k(pdl, k_order, 1, kScanThreads, st, a.atom_off, a.n_struct, a.order);
        return;
    }
    launch_k(pdl, k_order_parts, nch, kScanThreads, st, a.atom_off, a.n_struct, a.oparts);
    launch_k(true, k_order_final, nch, kScanThreads, st, a.atom_off, a.n_struct, (const int*)a.oparts, a.order);
}

size_t order_parts_bytes(int64_t n)
{
    const int64_t nch = (n + kScanItems * kScanThreads - 1) / (kScanItems * kScanThreads);
    return nch > 2 ? (size_t)4 * kOrderBins * nch : 0;
}

// CTAs of the enumeration: what fits on the SMs at once, or fewer where one item per warp would leave CTAs without one.
// A sphere has fewer parts than reflections; a shell's are estimated by those of the sphere that it is the rim of. Idle
// CTAs hold back the structure factor's, which then share SMs (one small cell in FP64 86 us a call, 102 with CTAs for all
// the parts that there is room for).
static int enum_grid(const GeomArgs& a, const void* kernel, size_t smem)
{
    const int nt = a.enum_threads;
    const int per_sm = resident_ctas(kernel, nt, smem);
    double parts = a.part_cap;
    if (a.cap_refl) parts = std::min(parts, (double)a.cap_refl / std::max(1.0 - std::pow(a.r2min / a.r2max, 1.5), 1e-12));
    const int64_t most = (a.n_struct + (int64_t)parts + nt / 32 - 1) / (nt / 32);
    return (int)std::min<int64_t>((int64_t)a.sms * per_sm, std::max<int64_t>(most, 1));
}

static ScanArgs scan_args(const GeomArgs& a)
{
    return ScanArgs{a.run_cnt, a.runs_mode ? 0 : 32 * a.rb, a.cap_refl, a.refl_off, a.tile_off, a.order, a.cls_list,
                    a.abort_flag, a.totals, a.status, a.work, a.aorder, a.atoms_set_geo ? a.atom_bad : nullptr, nullptr};
}

static void count_launch(const GeomArgs& a, const ScanArgs& sa, cudaStream_t st, bool pdl, bool last)
{
    const auto k = a.runs_mode ? k_count<true> : k_count<false>;
    const size_t smem = last && !sa.sums ? sizeof(long long) * kScanItems * (size_t)a.enum_threads : 0;
    const int grid = enum_grid(a, (const void*)k, smem);
    auto go = [&](auto launch) {
        launch(a.geo, a.n_struct, a.r2min, a.r2max, (float)a.r2min, (float)a.r2max, a.refl_cnt,
               a.run_cnt, a.enum_ctr, (const unsigned long long*)(a.enum_ctr + kPartCtr), (const int2*)a.part_tab, a.part_cnt,
               a.part_cap, enum_part_cols(a.n_struct, a.part_cap), sa, last ? a.enum_ctr + kDoneCtr : (int*)nullptr, sa.bad);
    };
    if (pdl) go([&](auto... v) { launch_pdl(k, grid, a.enum_threads, smem, st, v...); });
    else go([&](auto... v) { k<<<grid, a.enum_threads, smem, st>>>(v...); });
}

void launch_count_only(const GeomArgs& a, unsigned long long* sums, int tile_refl, cudaStream_t st)
{
    if (a.n_struct <= 0) return;
    prep_launch(false, a, st);
    ScanArgs sa{};
    sa.sums = sums;
    sa.tile_refl = tile_refl;
    count_launch(a, sa, st, true, sums != nullptr);
}

void launch_count(const GeomArgs& a, cudaStream_t st, bool pdl, bool scan)
{
    if (a.n_struct <= 0) return;
    ScanArgs sa = scan_args(a);
    if (!scan) sa.bad = nullptr;  // k_atoms has marked them
    count_launch(a, sa, st, pdl, scan);
}

int scan_chunks(int n) { return (n + kScanItems * kScanThreads - 1) / (kScanItems * kScanThreads); }

void launch_scan_refl(const GeomArgs& a, cudaStream_t st, bool pdl)
{
    const int nch = scan_chunks(a.n_struct);
    const int tile_refl = a.runs_mode ? 0 : 32 * a.rb;
    if (nch <= 2 || !a.parts) {  // one block walks the chunks
        launch_k(pdl, k_scan_refl, 1, kScanThreads, st, a.refl_cnt, a.geo, a.n_struct, scan_args(a));
        return;
    }
    launch_k(pdl, k_scan_refl_parts, nch, kScanThreads, st, a.refl_cnt, a.run_cnt, a.geo, a.n_struct, tile_refl,
             (const int*)a.order, a.parts, a.aorder ? a.oparts : (int*)nullptr);
    launch_k(true, k_scan_refl_final, nch, kScanThreads, st, a.refl_cnt, a.run_cnt, a.geo, a.n_struct, tile_refl,
             a.cap_refl, a.refl_off, a.tile_off, (const int*)a.order, a.cls_list, a.abort_flag, a.totals, a.status,
             a.work, (const long long*)a.parts, (const int*)a.oparts, a.aorder);
}

void launch_emit(const GeomArgs& a, cudaStream_t st, bool pdl)
{
    if (a.n_struct <= 0) return;
    const auto k = a.runs_mode ? k_emit<true> : k_emit<false>;
    const size_t smem = sizeof(ColRec) * (size_t)a.enum_threads;
    const int grid = enum_grid(a, (const void*)k, smem);
    auto go = [&](auto launch) {
        launch(a.geo, a.n_struct, a.r2min, a.r2max, (float)a.r2min, (float)a.r2max, 32 * a.rb,
               (const int64_t*)a.refl_off, (const int64_t*)a.run_cnt, (const int*)a.abort_flag, a.q, a.key, a.runs,
               (const int*)a.tile_off, a.tile_tab, a.enum_ctr + 1, (const unsigned long long*)(a.enum_ctr + kPartCtr),
               (const int2*)a.part_tab, (const int2*)a.part_cnt, a.part_cap, enum_part_cols(a.n_struct, a.part_cap));
    };
    if (pdl) go([&](auto... v) { launch_pdl(k, grid, a.enum_threads, smem, st, v...); });
    else go([&](auto... v) { k<<<grid, a.enum_threads, smem, st>>>(v...); });
}

}  // namespace xrd
