// Steps S2-S3: per-reflection scalars, structure factor and intensity.
//
// Sec. 2: per reflection, the sum of the atoms' contributions (the structure
// factor), corrected by the Lorentz-polarisation and Debye-Waller factors:
//   F(g) = sum_j occ_j f_j(s) exp(-B_j s^2) exp(2 pi i (h x_j + k y_j + l z_j)),
//   f(s) = Z - 41.78214 s^2 sum_i a_i exp(-b_i s^2),  s = |g| / 2,
//   I = |F|^2 (1 + cos^2 2theta) / (sin^2 theta cos theta),  sin theta = lambda |g| / 2.
//
// GB300 mapping: every warp of a persistent grid takes 128-reflection tiles of
// one structure (four reflections per lane) from an atomic queue in
// largest-first order. The warp stages the structure's atoms in shared memory
// and every lane walks the same atom list (one broadcast read per atom feeds
// four terms). Atoms are sorted by
// element, so f(s) is evaluated once per element run (a warp-uniform branch).
// The pattern variants form sin/cos on the FMA pipe from the exact phase
// (sincos_turn32) and use the SFU for exp2 (MUFU.EX2); the gradient variant
// uses the SFU for sin/cos too (MUFU.SIN/COS). FP64 arithmetic runs at
// about 1/64 of the FP32 rate here, so the phase is formed and reduced mod 1 in integers: from coordinates in 32-bit
// fixed point (XRD_FP32_PHASEFIX), or in 53-bit fixed point, the resolution of an FP64 phase (XRD_FP32_PHASE64: three
// more integer products a term; formed in FP64, four operations a term at 1.7 a clock and SM, it made the kernel take
// 471 us on 1024 cells of 1 to 64 atoms; now about 75 us; next to a rounding tie the FP64 phase is formed after all, so
// that the results are the same bits). The XRD_FP64 variant is k_sf64.cu.
#include <climits>

#include "xrd_internal.cuh"
#include "xrd_launch.h"

namespace xrd {

constexpr float kTwoPiOver2p32 = 1.4629180792671596e-09f;  // 2 pi / 2^32

// Launch shapes (chosen by xrd_autotune; default RB = 4, 2 warps per CTA):
// RB reflections per lane (one atom record feeds RB terms; tile = 32 RB
// reflections per warp) and WARPS warps per CTA.
constexpr int kSfChunk = 128;  // atoms staged per warp at a time

// Packed pairs of FP32 operations (FFMA2, FMUL2, FADD2): two reflections per instruction, each half rounded as the
// scalar operation rounds it.
__device__ __forceinline__ float2 dup2(float x) { return make_float2(x, x); }
__device__ __forceinline__ float2 ex2_2(float2 x) { return make_float2(ex2_approx(x.x), ex2_approx(x.y)); }
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return __ffma2_rn(b, dup2(-1.f), a); }  // a - b, one rounding

// Coef32 with every value twice, the operands of packed operations (64 bytes, shared memory)
struct __align__(16) CoefPair {
    float2 a[4];
    float2 bl[4];
};

// Atom32 as the loop reads it: (-B log2 e) and log2(occ) twice each
struct __align__(16) AtomPair {
    uint32_t X, Y, Z;
    int32_t z;
    float2 nb, lo;
};
__device__ __forceinline__ AtomPair atom_pair(const Atom32& a) { return AtomPair{a.X, a.Y, a.Z, a.z, dup2(a.nb), dup2(a.lo)}; }

__device__ __forceinline__ float2 f_of(const CoefPair& c, float2 zf, float2 s2)
{
    const float2 e0 = ex2_2(__fmul2_rn(c.bl[0], s2)), e1 = ex2_2(__fmul2_rn(c.bl[1], s2));
    const float2 e2 = ex2_2(__fmul2_rn(c.bl[2], s2)), e3 = ex2_2(__fmul2_rn(c.bl[3], s2));
    return __ffma2_rn(s2, __ffma2_rn(c.a[0], e0, __ffma2_rn(c.a[1], e1, __ffma2_rn(c.a[2], e2, __fmul2_rn(c.a[3], e3)))),
                      zf);
}

// sin and cos of two phases in turns (t: phase plus an eighth of a turn), the polynomials packed
__device__ __forceinline__ void sincos2_turn32(uint32_t t0, uint32_t t1, float2& s, float2& c)
{
    const float2 a = __fmul2_rn(make_float2(turn_rest(t0), turn_rest(t1)), dup2(kTurnScale));
    const float2 a2 = __fmul2_rn(a, a);
    const float2 ps = __ffma2_rn(__ffma2_rn(dup2(kSinC[2]), a2, dup2(kSinC[1])), a2, dup2(kSinC[0]));
    const float2 sa = __ffma2_rn(__fmul2_rn(a, a2), ps, a);
    const float2 pc =
        __ffma2_rn(__ffma2_rn(__ffma2_rn(dup2(kCosC[3]), a2, dup2(kCosC[2])), a2, dup2(kCosC[1])), a2, dup2(kCosC[0]));
    const float2 ca = __ffma2_rn(a2, pc, dup2(1.f));
    turn_quadrant(t0, sa.x, ca.x, s.x, c.x);
    turn_quadrant(t1, sa.y, ca.y, s.y, c.y);
}

__device__ __forceinline__ void sincos_turn32(uint32_t t, float& s, float& c)
{
    const float a = turn_rest(t) * kTurnScale, a2 = a * a;
    const float ps = fmaf(fmaf(kSinC[2], a2, kSinC[1]), a2, kSinC[0]);
    const float sa = fmaf(a * a2, ps, a);
    const float pc = fmaf(fmaf(fmaf(kCosC[3], a2, kCosC[2]), a2, kCosC[1]), a2, kCosC[0]);
    const float ca = fmaf(a2, pc, 1.f);
    turn_quadrant(t, sa, ca, s, c);
}

// Lorentz-polarisation factor (1 + cos^2 2theta) / (sin^2 theta cos theta) with
// sin^2 theta = X = q lambda^2 / 4. Up to 2theta = 90 degrees (X <= 1/2) the FP32
// cos^2 theta = 1 - X is good to a few ulp; above, its relative error grows as
// 1 / cos^2 theta (about 1.6e-5 at 170 degrees), so it is formed from |g|^2 in
// FP64 there (q: the reflection's |g|^2).
__device__ __forceinline__ float lp_of(float qf, float l2, const double* q, double lambda)
{
    const float X = qf * l2;  // sin^2 theta
    float u = 1.f - X;        // cos^2 theta
    if (X > 0.5f) u = fmaxf((float)fma(-0.25 * lambda * lambda, *q, 1.0), (float)kCos90Sq);
    const float c2 = fmaf(-2.f, X, 1.f);
    return fmaf(c2, c2, 1.f) / (X * sqrtf(u));
}

// d f / d s^2 = -41.78214 sum_i a_i exp(-b_i s^2)(1 - b_i s^2); with b_i = -bl_i ln 2
__device__ __forceinline__ float2 fprime_of(const CoefPair& c, float2 s2)
{
    const float2 ln2 = dup2(0.69314718055994531f);
    float2 acc = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < 4; i++)
        acc = __ffma2_rn(__fmul2_rn(c.a[i], ex2_2(__fmul2_rn(c.bl[i], s2))),
                         __ffma2_rn(__fmul2_rn(c.bl[i], ln2), s2, dup2(1.f)), acc);
    return acc;
}

// Signed low word of a 64-bit fixed-point coordinate, rounded to its upper 21 bits: with |h| <= 511 the sum of
// three index times low-word products stays below 2^31.
__device__ __forceinline__ int low21(int32_t lo) { return (lo >> 11) + ((lo >> 10) & 1); }

// The phase of XRD_FP32_PHASE64 is that of an FP64 evaluation, rounded to 2^-32 turns. The integer one errs by at most
// 0.501 (|h| + |k| + |l|) in units of 2^-53 (the coordinates' rounding), the FP64 one by half an ulp of each of three
// results, none above (|h| + |k| + |l|) times the largest coordinate. So both round alike unless the integer one is
// within phase_margin times |h| + |k| + |l| of a tie (one term in 10^4), where the FP64 one is formed.
__device__ __forceinline__ uint32_t phase_fp64(int h, int k, int l, const double* x)
{
    return fix32(fma((double)h, x[0], fma((double)k, x[1], (double)l * x[2])));
}
__device__ __forceinline__ int phase_margin(const double* x)
{
    const float m = fmaxf(fmaxf(__double2float_ru(fabs(x[0])), __double2float_ru(fabs(x[1]))), __double2float_ru(fabs(x[2])));
    return (int)fminf(4.1f * fmaxf(m, 1.f) + 1.f, 1048576.f);
}

// x / d correctly rounded, inv = 1 / d correctly rounded: Markstein's theorem (IBM J. Res. Dev. 34, 1990) makes one FMA
// step from a quotient within an ulp the rounded one; the first step gets it there. Five FP64 operations.
__device__ __forceinline__ double div_by(double x, double d, double inv)
{
    const double q0 = __dmul_rn(x, inv);
    const double q1 = __fma_rn(__fma_rn(-q0, d, x), inv, q0);
    return __fma_rn(__fma_rn(-q1, d, x), inv, q1);
}

// Grid cell b of 2theta and the position d within it, for the broadened profile (b = INT_MIN: no grid point within the
// window). In this kernel, whose FP64 unit is idle.
__device__ __forceinline__ void place(const CellArgs& c, int64_t r, double q)
{
    const double T = two_theta_q(q, c.l2h, c.l2l, c.ttab);
    const double pos = div_by(T - c.t0, c.dt, c.inv_dt);
    const double fb = floor(pos);
    const bool off = fb < (double)(-c.W - 1) || fb > (double)(c.n_pts + c.W);
    c.tb[r] = off ? INT_MIN : (int)fb;
    c.td[r] = off ? 0.f : (float)(pos - fb);
}

// The reflections of one lane in a tile: RUNS: one run of `len` reflections
// consecutive in l from `first` (step 1); otherwise up to RB reflections from
// `first` with a step of 32 (a tile of 32 RB consecutive reflections), `len` of
// them inside the structure.
//
// FP32 variants: every atom record (staged by the warp in shared memory, read
// by all lanes as a broadcast) feeds the lane's RB terms. With the integer phase
// (XRD_FP32_PHASEFIX) and RUNS, the phase factor is formed exactly once per run
// and atom, rotated from l to l + 1 by the atom's exp(2 pi i z) (an accurately
// rounded FP32 pair), and carried to l + 2 and l + 3 by the two-term recurrence
// e^{i(k+1)t} = 2 cos t e^{ikt} - e^{i(k-1)t} (two operations instead of four;
// rounding grows by a few ulp over a run of four): one sin/cos pair per run
// instead of per reflection. Otherwise every reflection's phase is formed exactly (integer
// phase; XRD_FP32_PHASE64 with the coordinates' low words too).
//
// The kernel is bound by instruction issue (about 77 % of the slots at 3 instructions a clock), so the FP32 work of two
// reflections goes into one packed instruction wherever both halves are at hand: the polynomials of sin and cos, f(s),
// the displacement factor's argument, the weights and the sums. The packed operations round each half as the scalar
// ones do: the results are the same bits. 256 cells of 200-2000 atoms: 10.20 -> 9.11 ms with runs; 100 000 mixed
// cells: 3.15 -> 2.85 ms. Fewer instructions alone do not make it faster: one packed sin/cos for two atoms of a run
// costs the moves that it saves (2.99 ms), and with a branch of its own for equal elements 9 % fewer instructions ran
// at 72 % (9.14 and 3.04 ms).
//
// Pattern variants (not GRAD): sin and cos come from the FMA pipe
// (sincos_turn32, five times more accurate than the SFU's), F is summed in FP32
// over blocks of 8 atoms (16 with runs) and
// each block sum is added into a two-float total (Knuth's TwoSum), so the
// rounding of the sum grows with the block size instead of the atom count
// (plain FP32 summation over N atoms errs by about 2e-8 sqrt(N) of the terms'
// root-sum-square). The lane also sums a_j^2, a_j = occ_j exp(-B_j s^2)
// max(|f_j|, Z_j), the scale of each term's rounding error (f_j itself may
// cancel to near zero; its rounding does not), and stores it for the
// re-evaluation of weak reflections (k_refine); with runs, once per run (its
// reflections, consecutive in l, have nearly equal s^2). Returns the lane's
// largest I.
// GRAD also accumulates dF/ds^2 = sum_j occ_j exp(-B_j s^2)(f_j' - B_j f_j) e^{i phi_j}.
template <int PREC, bool GRAD, int kSfRB, bool RUNS>
__device__ float sf_tile_fp32(const SfArgs& a, int s, int64_t first, int len, int64_t j0, int64_t j1, AtomPair* sat,
                              float2* sstep, int4* slo, const CoefPair* scoef, bool staged)
{
    constexpr float ln2 = 0.69314718055994531f;
    constexpr int step = RUNS ? 1 : 32;
    constexpr bool ACC = !GRAD;  // blocked two-float sum and the error scale
    constexpr int NP = kSfRB / 2;  // pairs of reflections
    const int lane = threadIdx.x & 31;
    float2 s2[NP], Fr[NP], Fi[NP], f[NP];
    float2 Gr[NP], Gi[NP], fp[NP];
    float2 Rh[NP], Rl[NP], Ih[NP], Il[NP], A2[NP];
    uint32_t uh[kSfRB], uk[kSfRB], ul[kSfRB];
    const float2 zero = make_float2(0.f, 0.f);
#pragma unroll
    for (int i = 0; i < kSfRB; i++) {
        const int64_t r = first + (int64_t)step * (i < len ? i : 0);
        const float v = d2f_pos(a.q[r]) * 0.25f;
        if (i & 1) s2[i / 2].y = v;
        else s2[i / 2].x = v;
        if (!RUNS || i == 0) {
            const uint32_t key = a.key[r];
            uh[i] = (uint32_t)hkl_h(key); uk[i] = (uint32_t)hkl_k(key); ul[i] = (uint32_t)hkl_l(key);
        } else {
            uh[i] = uh[0]; uk[i] = uk[0]; ul[i] = ul[0] + (uint32_t)i;
        }
    }
#pragma unroll
    for (int p = 0; p < NP; p++) Fr[p] = Fi[p] = f[p] = Gr[p] = Gi[p] = fp[p] = Rh[p] = Rl[p] = Ih[p] = Il[p] = A2[p] = zero;
    float zf = 0.f, fm = 0.f;  // fm, with runs: max(|f|, Z) of the first reflection
    constexpr bool kRotate = RUNS && PREC == XRD_FP32_PHASEFIX;
    constexpr int kFold = kRotate ? 16 : 8;  // block size of the two-float sum: 16 atoms with runs, else 8
    int zc = -1;
    int hkl1 = 0;  // the largest |h| + |k| + |l| of the lane's reflections
    if (PREC == XRD_FP32_PHASE64)
#pragma unroll
        for (int i = 0; i < kSfRB; i++) hkl1 = max(hkl1, abs((int)uh[i]) + abs((int)uk[i]) + abs((int)ul[i]));
    for (int64_t c0 = j0; c0 < j1; c0 += kSfChunk) {
        const int nc = (int)min((int64_t)kSfChunk, j1 - c0);
        if (!staged) {
            __syncwarp();
            for (int i = lane; i < nc; i += 32) {
                AtomPair at = atom_pair(a.atom32[c0 + i]);
                if (kRotate) sstep[i] = a.astep[c0 + i];
                if (PREC == XRD_FP32_PHASE64) {
                    const AtomX d = a.atomx[c0 + i];
                    at.X = d.hi[0];
                    at.Y = d.hi[1];
                    at.Z = d.hi[2];
                    slo[i] = make_int4(low21(d.lo[0]), low21(d.lo[1]), low21(d.lo[2]),
                                       phase_margin(a.frac + 3 * (j0 + a.atom32[c0 + i].src)));
                }
                sat[i] = at;
            }
            __syncwarp();
        }
        for (int jb = 0; jb < nc; jb += kFold) {
            const int je = min(jb + kFold, nc);
#pragma unroll 1
            for (int jj = jb; jj < je; jj++) {
                const AtomPair at = sat[jj];
                if (at.z != zc) {  // uniform: every lane walks the same element-sorted list
                    zc = at.z;
                    zf = (float)zc;
                    const CoefPair c = scoef[zc];
#pragma unroll
                    for (int p = 0; p < NP; p++) {
                        f[p] = f_of(c, dup2(zf), s2[p]);
                        if (GRAD) fp[p] = fprime_of(c, s2[p]);
                        if (kRotate && p == 0) fm = fmaxf(fabsf(f[0].x), zf);
                    }
                }
                float2 cs[NP], sn[NP];
                if (kRotate) {  // the run's phase factors from its first one
                    float s0, co;
                    sincos_turn32(uh[0] * at.X + kEighthTurn + uk[0] * at.Y + ul[0] * at.Z, s0, co);
                    const float2 st = sstep[jj];
                    const float tcz = st.x + st.x;  // exact
                    cs[0].x = co;
                    sn[0].x = s0;
                    // the rotation by exp(2 pi i z), then e^{i(k+1)t} = 2 cos t e^{ikt} - e^{i(k-1)t}
                    cs[0].y = fmaf(co, st.x, -s0 * st.y);
                    sn[0].y = fmaf(co, st.y, s0 * st.x);
#pragma unroll
                    for (int p = 1; p < NP; p++) {
                        cs[p].x = fmaf(tcz, cs[p - 1].y, -cs[p - 1].x);
                        sn[p].x = fmaf(tcz, sn[p - 1].y, -sn[p - 1].x);
                        cs[p].y = fmaf(tcz, cs[p].x, -cs[p - 1].y);
                        sn[p].y = fmaf(tcz, sn[p].x, -sn[p - 1].y);
                    }
                } else {
                    uint32_t P[kSfRB];
#pragma unroll
                    for (int i = 0; i < kSfRB; i++)
                        P[i] = uh[i] * at.X + (ACC ? kEighthTurn : 0u) + uk[i] * at.Y + ul[i] * at.Z;
                    if (PREC == XRD_FP32_PHASE64) {  // the low words' sums, below 2^31, rounded into the high words'
                        const int4 lo = slo[jj];
                        const uint32_t near = min((uint32_t)hkl1 * (uint32_t)lo.w + 2u, 1u << 20);
                        bool tie = false;
#pragma unroll
                        for (int i = 0; i < kSfRB; i++) {
                            const int v = (int)uh[i] * lo.x + (int)uk[i] * lo.y + (int)ul[i] * lo.z + (1 << 20);
                            P[i] += (uint32_t)(v >> 21);
                            tie |= (((uint32_t)v + near) & 0x1fffffu) <= 2u * near;
                        }
                        if (tie) {  // the FP64 phase may round the other way
                            const double* x = a.frac + 3 * (j0 + a.atom32[c0 + jj].src);
#pragma unroll
                            for (int i = 0; i < kSfRB; i++)
                                P[i] = phase_fp64((int)uh[i], (int)uk[i], (int)ul[i], x) + kEighthTurn;
                        }
                    }
#pragma unroll
                    for (int p = 0; p < NP; p++) {
                        if (ACC) {
                            sincos2_turn32(P[2 * p], P[2 * p + 1], sn[p], cs[p]);
                        } else {
                            __sincosf((float)(int32_t)P[2 * p] * kTwoPiOver2p32, &sn[p].x, &cs[p].x);
                            __sincosf((float)(int32_t)P[2 * p + 1] * kTwoPiOver2p32, &sn[p].y, &cs[p].y);
                        }
                    }
                }
#pragma unroll
                for (int p = 0; p < NP; p++) {
                    const float2 dw = ex2_2(__ffma2_rn(at.nb, s2[p], at.lo));
                    const float2 w = __fmul2_rn(f[p], dw);
                    Fr[p] = __ffma2_rn(w, cs[p], Fr[p]);
                    Fi[p] = __ffma2_rn(w, sn[p], Fi[p]);
                    if (ACC) {
                        if (kRotate) {  // a run's reflections share one scale (s^2 nearly equal)
                            if (p == 0) {
                                const float m = dw.x * fm;
                                A2[0].x = fmaf(m, m, A2[0].x);
                            }
                        } else {
                            const float2 m = __fmul2_rn(dw, make_float2(fmaxf(fabsf(f[p].x), zf), fmaxf(fabsf(f[p].y), zf)));
                            A2[p] = __ffma2_rn(m, m, A2[p]);
                        }
                    }
                    if (GRAD) {
                        const float2 wd = __fmul2_rn(__ffma2_rn(__fmul2_rn(at.nb, dup2(ln2)), f[p], fp[p]), dw);
                        Gr[p] = __ffma2_rn(wd, cs[p], Gr[p]);
                        Gi[p] = __ffma2_rn(wd, sn[p], Gi[p]);
                    }
                }
            }
            if (ACC) {  // block sums into the two-float totals
#pragma unroll
                for (int p = 0; p < NP; p++) {
                    float2 t = __fadd2_rn(Rh[p], Fr[p]), bb = sub2(t, Rh[p]);
                    Rl[p] = __fadd2_rn(Rl[p], __fadd2_rn(sub2(Rh[p], sub2(t, bb)), sub2(Fr[p], bb)));
                    Rh[p] = t;
                    t = __fadd2_rn(Ih[p], Fi[p]);
                    bb = sub2(t, Ih[p]);
                    Il[p] = __fadd2_rn(Il[p], __fadd2_rn(sub2(Ih[p], sub2(t, bb)), sub2(Fi[p], bb)));
                    Ih[p] = t;
                    Fr[p] = zero;
                    Fi[p] = zero;
                }
            }
        }
    }
    auto half = [](const float2* v, int i) { return i & 1 ? v[i / 2].y : v[i / 2].x; };
    const float l2 = a.l2f;
    float imax = 0.f;
#pragma unroll
    for (int i = 0; i < kSfRB; i++) {
        if (i >= len) continue;
        const int64_t r = first + (int64_t)step * i;
        const float qf = d2f_pos(a.q[r]);
        const float fr = ACC ? half(Rh, i) + half(Rl, i) : half(Fr, i);
        const float fi = ACC ? half(Ih, i) + half(Il, i) : half(Fi, i);
        const float F2 = fmaf(fr, fr, fi * fi), lp = lp_of(qf, l2, a.q + r, a.lambda);
        const float I = F2 * lp;
        if (GRAD) {
            a.Fx[r] = make_float4(fr, fi, half(Gr, i), half(Gi, i));
            a.Ig[r] = I;
            place(a.cell, r, a.q[r]);
        } else {
            a.If[r] = I;
            if (ACC && a.Eb) {
                // the bound of the rounding error of I; a reflection can need the re-evaluation only if
                // it exceeds tau of I (the criterion is E > tau max(I, c M)): then its structure is noted
                const float dF = a.eps_k * sqrtf(half(A2, kRotate ? 0 : i));
                const float E = lp * dF * fmaf(2.f, sqrtf(F2), dF);
                a.Eb[r] = E;
                if (E > a.tau * I) a.Es[r] = s;
            }
            if (a.F) a.F[r] = make_float2(fr, fi);
            imax = fmaxf(imax, I);
        }
    }
    return imax;
}

// Structures by reflection count, largest first (buckets of a quarter octave), by one CTA beside the tiles of the
// others: the profile kernels that follow give every structure a CTA and start with the largest. cnt: kCountBuckets
// ints of shared memory. The order within a bucket is arbitrary; nothing but the load balance depends on it. For the small
// batches of the one-launch front, where it ends before the tiles do; in the scan of the counts, which orders the others, it
// lengthened the chain of launches (1024 small cells 190.8 -> 194.4 us a call).
constexpr int kCountBuckets = 128;
__device__ void order_by_count(const SfArgs& a, int* cnt)
{
    for (int i = threadIdx.x; i < kCountBuckets; i += blockDim.x) cnt[i] = 0;
    __syncthreads();
    // f(s, bucket) of every structure, the counts of four read together
    auto each = [&](auto f) {
        for (int s0 = threadIdx.x; s0 < a.n_struct; s0 += 4 * blockDim.x) {
            int64_t R[4];
#pragma unroll
            for (int u = 0; u < 4; u++) {
                const int s = min(s0 + u * (int)blockDim.x, a.n_struct - 1);
                R[u] = a.refl_off[s + 1] - a.refl_off[s];
            }
#pragma unroll
            for (int u = 0; u < 4; u++)
                if (s0 + u * (int)blockDim.x < a.n_struct)
                    f(s0 + u * (int)blockDim.x, R[u] <= 0 ? 0 : min(kCountBuckets - 1, 1 + (int)(4.f * log2f((float)R[u]))));
        }
    };
    each([&](int, int b) { atomicAdd(&cnt[b], 1); });
    __syncthreads();
    if (threadIdx.x == 0) {
        int acc = 0;
        for (int b = kCountBuckets - 1; b >= 0; b--) {
            const int c = cnt[b];
            cnt[b] = acc;
            acc += c;
        }
    }
    __syncthreads();
    each([&](int s, int b) { a.aorder[atomicAdd(&cnt[b], 1)] = s; });
}

// Persistent CTAs; every warp takes tiles of 32 runs (one per lane) from a
// queue in largest-first order (tiles of the structures with the most atoms
// first). A structure's atoms stay staged in the warp's shared memory while its
// consecutive tiles follow (when they fit one chunk).
// Register caps: 64 for the integer-phase variant with 2 reflections per lane
// (32 resident warps per SM), 72 with runs (28 warps asked for, 26 fit beside the staged atoms: 2.85 ms on 100 000
// mixed cells, 2.88 with 24), about 85 for the other FP32 variants (24 warps).
template <int PREC, bool GRAD, int RB, int WARPS, bool RUNS>
__global__ void __launch_bounds__(32 * WARPS,
                                  (PREC == XRD_FP32_PHASEFIX && !GRAD && RB == 2) ? 32 / WARPS
                                  : (PREC == XRD_FP32_PHASE64 && RB == 4)         ? 20 / WARPS
                                                                                  : (RUNS ? 28 : 24) / WARPS)
    k_sf(const SfArgs a)
{
    pdl_enter();
    constexpr int kSfThreads = 32 * WARPS;
    __shared__ AtomPair sat[WARPS][kSfChunk];
    __shared__ float2 sstep[RUNS ? WARPS : 1][RUNS ? kSfChunk : 1];
    __shared__ int4 slo[PREC == XRD_FP32_PHASE64 ? WARPS : 1][PREC == XRD_FP32_PHASE64 ? kSfChunk : 1];
    extern __shared__ CoefPair scoef[];  // [zmax + 1]
    if (a.aorder && blockIdx.x == gridDim.x - 1) {
        __shared__ int cnt[kCountBuckets];
        order_by_count(a, cnt);
    }
    if (*a.abort_flag) return;
    const int ntiles = a.tile_off[a.n_struct];
    if ((int)blockIdx.x >= ntiles) return;  // the CTAs before this one already have a tile each
    for (int z = threadIdx.x; z <= a.zmax; z += kSfThreads) {
        const Coef32 c = a.coef32[z];
        for (int i = 0; i < 4; i++) {
            scoef[z].a[i] = dup2(c.a[i]);
            scoef[z].bl[i] = dup2(c.bl[i]);
        }
    }
    __syncthreads();
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    int staged_s = -1;  // structure whose atoms (one chunk at most) are in sat[w]
    for (;;) {
        int t = 0;
        if (lane == 0) t = atomicAdd(a.tile_counter, 1);
        t = __shfl_sync(0xffffffffu, t, 0);
        if (t >= ntiles) break;
        const int2 e = a.tile_tab[t];
        const int s = e.x;
        const int64_t rbase = a.refl_off[s], re = a.refl_off[s + 1];
        const int64_t j0 = a.atom_off[s], j1 = a.atom_off[s + 1];
        int64_t first;
        int len;
        if (RUNS) {  // lane: one run of the structure
            const int64_t nruns = a.run_cnt[s];
            const int64_t r = e.y + lane;
            int start = 0;
            len = 0;
            if (r < nruns) {
                const int pk = a.runs[rbase + r];
                start = pk >> 3;
                len = pk & 7;
            }
            first = rbase + start;
        } else {  // lane: reflections e.y + lane + 32 i of the structure
            first = rbase + e.y + lane;
            len = (int)max(min((re - first + 31) / 32, (int64_t)RB), (int64_t)0);
        }
        if (len == 0) first = rbase;  // keep the lane's (ignored) loads inside the array
        const bool one_chunk = j1 - j0 <= kSfChunk;
        float m = sf_tile_fp32<PREC, GRAD, RB, RUNS>(a, s, first, len, j0, j1, sat[w], sstep[RUNS ? w : 0],
                                                     slo[PREC == XRD_FP32_PHASE64 ? w : 0], scoef,
                                                     one_chunk && s == staged_s);
        staged_s = one_chunk ? s : -1;
        if (!GRAD && a.imax) {  // the structure's largest reflection intensity (I >= 0: integer order)
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
            if (lane == 0 && m > 0.f) atomicMax(a.imax + s, __float_as_uint(m));
        }
    }
}

template <int PREC, bool GRAD, int RB, int WARPS, bool RUNS>
static void launch_sf_shape(const SfArgs& a, cudaStream_t st, bool pdl)
{
    // persistent grid: as many CTAs as fit on the SMs at once (cached per device and zmax)
    static int cache_per_sm[64] = {}, cache_zmax[64] = {};
    const size_t smem = sizeof(CoefPair) * (size_t)(a.zmax + 1);
    int dev = 0;
    cudaGetDevice(&dev);
    const bool cached = dev >= 0 && dev < 64 && cache_per_sm[dev] > 0 && cache_zmax[dev] == a.zmax;
    int per_sm = cached ? cache_per_sm[dev] : 0;
    if (!cached) {
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sf<PREC, GRAD, RB, WARPS, RUNS>, 32 * WARPS,
                                                          smem) != cudaSuccess ||
            per_sm < 1)
            per_sm = 4;
        if (dev >= 0 && dev < 64) { cache_per_sm[dev] = per_sm; cache_zmax[dev] = a.zmax; }
    }
    if (pdl) launch_pdl(k_sf<PREC, GRAD, RB, WARPS, RUNS>, a.grid * per_sm, 32 * WARPS, smem, st, a);
    else k_sf<PREC, GRAD, RB, WARPS, RUNS><<<a.grid * per_sm, 32 * WARPS, smem, st>>>(a);
}

template <int PREC, bool GRAD>
static void launch_sf_prec(const SfArgs& a, cudaStream_t st, bool pdl)
{
    if (a.rb == 2) launch_sf_shape<PREC, GRAD, 2, 2, false>(a, st, pdl);
    else launch_sf_shape<PREC, GRAD, 4, 2, false>(a, st, pdl);
}

// a.grid = number of SMs; a.rb, a.warps, a.runs_mode = launch shape. Runs (with the l-step
// rotation) exist for the integer-phase pattern variant with 4 reflections per lane.
void launch_sf(const SfArgs& a, cudaStream_t st, bool pdl)
{
    if (a.n_struct <= 0) return;
    if (a.Fx) {  // gradient path: FP32 with the integer phase
        launch_sf_prec<XRD_FP32_PHASEFIX, true>(a, st, pdl);
        return;
    }
    switch (a.precision) {
    case XRD_FP64: launch_sf64(a, st, pdl); break;
    case XRD_FP32_PHASE64: launch_sf_prec<XRD_FP32_PHASE64, false>(a, st, pdl); break;
    default:
        if (a.runs_mode) {
            if (a.warps == 1) launch_sf_shape<XRD_FP32_PHASEFIX, false, 4, 1, true>(a, st, pdl);
            else if (a.warps == 4) launch_sf_shape<XRD_FP32_PHASEFIX, false, 4, 4, true>(a, st, pdl);
            else launch_sf_shape<XRD_FP32_PHASEFIX, false, 4, 2, true>(a, st, pdl);
        } else if (a.rb == 2) {
            if (a.warps == 1) launch_sf_shape<XRD_FP32_PHASEFIX, false, 2, 1, false>(a, st, pdl);
            else if (a.warps == 4) launch_sf_shape<XRD_FP32_PHASEFIX, false, 2, 4, false>(a, st, pdl);
            else launch_sf_shape<XRD_FP32_PHASEFIX, false, 2, 2, false>(a, st, pdl);
        } else {
            if (a.warps == 1) launch_sf_shape<XRD_FP32_PHASEFIX, false, 4, 1, false>(a, st, pdl);
            else if (a.warps == 4) launch_sf_shape<XRD_FP32_PHASEFIX, false, 4, 4, false>(a, st, pdl);
            else launch_sf_shape<XRD_FP32_PHASEFIX, false, 4, 2, false>(a, st, pdl);
        }
        break;
    }
}

}  // namespace xrd
