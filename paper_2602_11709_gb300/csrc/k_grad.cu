// Steps S7-S8: Gaussian-broadened pattern and its adjoint.
//
// The broadened profile y_k = sum_g I_g exp(-(t_k - 2theta_g)^2 / (2 sigma^2))
// is the differentiable form of the pattern used for refinement and for
// training patterns with peak broadening (Sec. 1). Each Friedel-unique
// reflection stands for g and -g (weight 2). Every Gaussian is cut to the grid
// points b - W .. b + W + 1 around its grid cell b, W = ceil(6 sigma / dt), in
// the forward and the backward pass alike, so the gradient is the exact
// gradient of the computed y.
//
// Adjoint, per reflection r (F, dF/ds^2 saved by the forward pass):
//   dL/dI_r = 2 sum_k g_k G_rk,  dL/d2theta_r = 2 I_r sum_k g_k G_rk (t_k - 2theta_r) / sigma^2,
//   dI/dx_j = 4 pi h LP w_j (Im F cos phi_j - Re F sin phi_j)   (likewise y with k, z with l),
//   dI/dB_j = -2 LP s^2 w_j (Re F cos phi_j + Im F sin phi_j),
//   dI/dq  = LP Re(conj F dF/ds^2) / 2 + |F|^2 dLP/dq,  q = |g|^2 = h^T G* h,
//   dL/dG* = sum_r dL/dq_r h h^T,  dL/dG = -G* (dL/dG*) G*,  then G(a, b, c, alpha, beta, gamma).
#include <cmath>

#include "xrd_internal.cuh"
#include "xrd_launch.h"

namespace xrd {

constexpr int kReflCluster = 4;
constexpr int kReflThreads = 128;

__device__ __forceinline__ void cluster_sync()
{
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// the 16 bytes at this CTA's shared address p in CTA `rank` of the cluster
__device__ __forceinline__ float4 cluster_load(const float4* p, int rank)
{
    uint32_t at = (uint32_t)__cvta_generic_to_shared(p), to;
    float4 v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(to) : "r"(at), "r"(rank));
    asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];"
                 : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
                 : "r"(to)
                 : "memory");
    return v;
}
__device__ __forceinline__ double cluster_load(const double* p, int rank)
{
    uint32_t at = (uint32_t)__cvta_generic_to_shared(p), to;
    double v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(to) : "r"(at), "r"(rank));
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(to) : "memory");
    return v;
}

// ---------------------------------------------------------------- forward: broadened pattern

// One CTA per structure, those with the most reflections first: the reflections sorted by grid cell (counting sort,
// each cell by index, so that the sums do
// not depend on the run), then every grid point sums its window. The sorted cell, offset and amplitude of each
// reflection are written once and read in order (through the permutation every term was a chain of two dependent
// loads). The cells themselves come from the structure-factor kernel, whose FP64 unit is free, where 13 FP64 operations
// a reflection bound this one. 512 cells of 8 to 128 atoms on 4096 points: 127 us with 256 threads a structure, the
// permutation and the cells formed here, 33 us now (and 6 us more in the structure-factor kernel).
// Threads: 1024 while the structures are few enough that the largest sets the time, up to kBroadenFew a SM; beyond,
// 512, since the short phases between barriers of more CTAs overlap (512 cells of 8-128 atoms on 4096 points 310 us a step
// with 1024 and 321 with 512; 1500 cells of 3 atoms on 257 points 286 and 258, 100 000 one-atom cells 6.5 and 5.9 ms).
constexpr int kBroadenMaxThreads = 1024;
constexpr int kBroadenFew = 4;

// PER consecutive points a thread, whose windows share most reflections where these are dense (16 cells of 200-2000 atoms
// on 4096 points 14.2 ms a step with four, 14.5 with one); on a grid of fewer points than that needs, four left most
// threads idle (3000 one-atom cells on 257 points 1.16 ms a step, 0.97 with one).
template <int PER>
__device__ __forceinline__ void broaden_gather(int n_pts, int W, float dt, float cg, const int* bins,
                                               const int* __restrict__ sb, const float2* __restrict__ sda,
                                               float* __restrict__ yo)
{
    for (int k0 = PER * threadIdx.x; k0 < n_pts; k0 += PER * blockDim.x) {
        float acc[PER];
        int lo[PER], hi[PER];
#pragma unroll
        for (int j = 0; j < PER; j++) {
            const int k = min(k0 + j, n_pts - 1);
            acc[j] = 0.f;
            lo[j] = k ? bins[k - 1] : 0;
            hi[j] = bins[k + 2 * W + 1];  // cells c = b + W + 1 of k .. k + 2 W + 1
        }
        for (int i = lo[0]; i < hi[PER - 1]; i++) {
            const float2 v = sda[i];
            const int b = sb[i];
#pragma unroll
            for (int j = 0; j < PER; j++) {
                const float u = ((float)(k0 + j - b) - v.x) * dt;
                const float t = fmaf(v.y, ex2_approx(-u * u * cg), acc[j]);
                if (i >= lo[j] && i < hi[j]) acc[j] = t;
            }
        }
#pragma unroll
        for (int j = 0; j < PER; j++)
            if (k0 + j < n_pts) yo[k0 + j] = acc[j];
    }
}

__global__ void __launch_bounds__(kBroadenMaxThreads) k_broaden(const GradArgs a)
{
    pdl_enter();
    extern __shared__ int bins[];  // cell counts, then offsets; cells c = b + W + 1 in [0, nb)
    __shared__ int tmp[34];
    const int s = a.aorder[blockIdx.x];  // the structures with the most reflections first
    float* __restrict__ yo = a.y + (int64_t)s * a.n_pts;
    if (*a.abort_flag) {
        for (int k = threadIdx.x; k < a.n_pts; k += blockDim.x) yo[k] = 0.f;
        return;
    }
    const int64_t base = a.refl_off[s];
    const int n = (int)(a.refl_off[s + 1] - base);
    const int W = a.W, nb = a.n_pts + 2 * W + 2;
    const float cg = a.cg;
    for (int c = threadIdx.x; c <= nb; c += blockDim.x) bins[c] = 0;
    __syncthreads();
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const int b = a.tb[base + i];
        if (b != INT_MIN) atomicAdd(&bins[b + W + 1], 1);
    }
    __syncthreads();
    block_excl_scan(bins, nb, tmp);
    __syncthreads();
    int* __restrict__ perm = a.perm + base;
    for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const int b = a.tb[base + i];
        if (b != INT_MIN) perm[atomicAdd(&bins[b + W + 1], 1)] = i;
    }
    __syncthreads();
    // bins[c] is now the end of cell c; order each cell by reflection index (deterministic sums)
    for (int c = threadIdx.x; c < nb; c += blockDim.x) {
        const int c0 = c ? bins[c - 1] : 0, c1 = bins[c];
        for (int i = c0 + 1; i < c1; i++) {
            const int v = perm[i];
            int j = i - 1;
            while (j >= c0 && perm[j] > v) {
                perm[j + 1] = perm[j];
                j--;
            }
            perm[j + 1] = v;
        }
    }
    __syncthreads();
    const int nin = nb ? bins[nb - 1] : 0;  // reflections with a window on the grid
    int* __restrict__ sb = a.sb + base;
    float2* __restrict__ sda = a.sda + base;
    for (int i = threadIdx.x; i < nin; i += blockDim.x) {
        const int64_t r = base + perm[i];
        sb[i] = a.tb[r];
        sda[i] = make_float2(a.td[r], 2.f * a.Ig[r]);
    }
    __syncthreads();
    // gather: grid point k sees the reflections of cells b in [k - W - 1, k + W]
    const float dt = (float)a.dt;
    if (a.n_pts >= 4 * (int)blockDim.x) broaden_gather<4>(a.n_pts, W, dt, cg, bins, sb, sda, yo);
    else broaden_gather<1>(a.n_pts, W, dt, cg, bins, sb, sda, yo);
}

// ---------------------------------------------------------------- backward: per reflection + lattice

// d G / d p of one lattice parameter (p = 0 .. 5) contracted with the symmetric DG (elements 11, 22, 33, 12, 13, 23)
__device__ __forceinline__ double dL_dp(const double* DG, const double* lat, int p, double ca, double cb, double cg,
                                        double sn)
{
    const double a = lat[0], b = lat[1], c = lat[2], rad = kPi / 180.0;
    switch (p) {
    case 0: return 2 * a * DG[0] + 2 * (b * cg * DG[3] + c * cb * DG[4]);
    case 1: return 2 * b * DG[1] + 2 * (a * cg * DG[3] + c * ca * DG[5]);
    case 2: return 2 * c * DG[2] + 2 * (a * cb * DG[4] + b * ca * DG[5]);
    case 3: return -2 * b * c * sn * rad * DG[5];
    case 4: return -2 * a * c * sn * rad * DG[4];
    default: return -2 * a * b * sn * rad * DG[3];
    }
}

// A cluster of kReflCluster CTAs per structure, those with the most reflections first: one CTA a structure left the
// largest (three times the mean) to a few SMs, where its FP64 sums queue for the unit. 512 cells of 8 to 128 atoms: 80 us
// with a CTA a structure and one thread for the lattice, 43 us now.
__global__ void __launch_bounds__(kReflThreads) k_grad_refl(const GradArgs a)
{
    pdl_enter();
    __shared__ double part[6][kReflThreads], red[6];
    const int s = a.aorder[blockIdx.x / kReflCluster], rank = blockIdx.x % kReflCluster;  // the cluster is a row of the grid
    const bool ok = !*a.abort_flag && a.geo[s].status == XRD_OK;
    const int64_t base = a.refl_off[s];
    const int n = ok ? (int)(a.refl_off[s + 1] - base) : 0;
    const int W = a.W;
    const float cg = a.cg, inv_s2 = a.inv_s2;
    const float dt = (float)a.dt, l2 = (float)a.l2d;
    const float* __restrict__ g = a.dLdy + (int64_t)s * a.n_pts;
    double m6[6] = {0, 0, 0, 0, 0, 0};
    for (int i = rank * kReflThreads + (int)threadIdx.x; i < n; i += kReflCluster * kReflThreads) {
        const int64_t r = base + i;
        const int b = a.tb[r];
        float sI = 0.f, sT = 0.f;
        if (b != INT_MIN) {
            const float d = a.td[r];
            const int k0 = max(0, b - W), k1 = min(a.n_pts - 1, b + W + 1);
            for (int k = k0; k <= k1; k++) {
                const float u = ((float)(k - b) - d) * dt;
                const float G = ex2_approx(-u * u * cg);
                sI = fmaf(g[k], G, sI);
                sT = fmaf(g[k] * G, u, sT);
            }
        }
        const float4 F = a.Fx[r];
        const float I = a.Ig[r];
        const float dLdI = 2.f * sI;
        const float dLdT = 2.f * I * sT * inv_s2;
        const double qd = a.q[r];
        const float qf = d2f_pos(qd);
        const float X = qf * l2;  // sin^2 theta
        float cc = 1.f - X;       // cos^2 theta; above 2theta = 90 degrees from |g|^2 in FP64 (cancellation)
        if (X > 0.5f) cc = fmaxf((float)fma(-a.l2d, qd, 1.0), (float)kCos90Sq);
        const float c2 = fmaf(-2.f, X, 1.f), rt = sqrtf(cc);
        const float N = fmaf(c2, c2, 1.f), D = X * rt;
        const float lp = N / D;
        const float dlp = (-4.f * c2 * D - N * (rt - X / (2.f * rt))) / (D * D) * l2;
        const float dT = (float)(360.0 / kPi) / (2.f * sqrtf(X) * rt) * l2;
        const float alpha = dLdI * lp;
        a.U[r] = alpha * F.x;
        a.V[r] = alpha * F.y;
        const float FF = fmaf(F.x, F.x, F.y * F.y);
        const float dIdq = fmaf(0.5f * lp, fmaf(F.x, F.z, F.y * F.w), FF * dlp);
        const double wq = f2d_fast(fmaf(dLdI, dIdq, dLdT * dT));
        const uint32_t key = a.key[r];
        const int h = hkl_h(key), k = hkl_k(key), l = hkl_l(key);
        m6[0] = fma(wq, i2d_exact(h * h), m6[0]);
        m6[1] = fma(wq, i2d_exact(k * k), m6[1]);
        m6[2] = fma(wq, i2d_exact(l * l), m6[2]);
        m6[3] = fma(wq, i2d_exact(h * k), m6[3]);
        m6[4] = fma(wq, i2d_exact(h * l), m6[4]);
        m6[5] = fma(wq, i2d_exact(k * l), m6[5]);
    }
    // deterministic reduction of the six sums: in the CTA (a shuffle reduction of every sum in every warp takes three
    // times the FP64 additions), then over the cluster
    const int w = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int c = 0; c < 6; c++) part[c][threadIdx.x] = m6[c];
    __syncthreads();
    for (int c = w; c < 6; c += kReflThreads / 32) {
        double v = part[c][lane];
        for (int i = 1; i < kReflThreads / 32; i++) v += part[c][lane + 32 * i];
        for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
        if (lane == 0) red[c] = v;
    }
    cluster_sync();
    double t = 0.0;
    if (rank == 0 && w == 0 && lane < 6)
        for (int r = 0; r < kReflCluster; r++) t += cluster_load(&red[lane], r);
    cluster_sync();  // read before the other CTAs end
    if (rank != 0 || w != 0) return;
    // One warp, a lane per value, ends it: FP64 runs at 1.7 operations a clock and SM with a long latency, and one
    // thread's 24 cosines and sines took most of the kernel.
    float* __restrict__ out = a.d_lat + 6 * (int64_t)s;
    if (!ok) {
        if (lane < 6) out[lane] = 0.f;
        return;
    }
    const double* lat = a.lattice + 6 * (int64_t)s;
    double sn = 0.0, cs = 0.0;
    if (lane >= 3 && lane < 6) sincos(lat[lane] * (kPi / 180.0), &sn, &cs);
    const double ca = __shfl_sync(0xffffffffu, cs, 3), cb = __shfl_sync(0xffffffffu, cs, 4),
                 cgm = __shfl_sync(0xffffffffu, cs, 5);
    // dL/dG* as a full symmetric matrix (q = sum over all a, b of G*_ab h_a h_b); lanes 0 to 8 hold its elements (i, j)
    const int i = lane / 3, j = lane % 3;
    auto sym = [](int x, int y) { return x == y ? x : x + y + 2; };  // (11, 22, 33, 12, 13, 23)
    const double M = __shfl_sync(0xffffffffu, t, lane < 9 ? sym(i, j) : 0);
    const double* gs = a.geo[s].gs;
    const double S = lane < 9 ? gs[sym(i, j)] : 0.0;
    double SM = 0.0, DG = 0.0;  // dL/dG = -G* (dL/dG*) G*
    for (int m = 0; m < 3; m++)
        SM += __shfl_sync(0xffffffffu, S, (3 * i + m) & 31) * __shfl_sync(0xffffffffu, M, (3 * m + j) & 31);
    for (int m = 0; m < 3; m++)
        DG -= __shfl_sync(0xffffffffu, SM, (3 * i + m) & 31) * __shfl_sync(0xffffffffu, S, (3 * m + j) & 31);
    double D6[6];
    const int at[6] = {0, 4, 8, 1, 2, 5};
    for (int e = 0; e < 6; e++) D6[e] = __shfl_sync(0xffffffffu, DG, at[e]);
    if (lane < 6) out[lane] = (float)dL_dp(D6, lat, lane, ca, cb, cgm, sn);
}

// ---------------------------------------------------------------- backward: atoms

// A cluster of kAtomCluster CTAs per structure, the structures with the most atoms first; each CTA holds 64 of the
// structure's 256 sums, four warps for each 32 of them, a lane a sum. Sum t belongs to atom t mod Nc of the current atom chunk and every P-th
// reflection (residue t / Nc) of each kAtomChunkRefl, added in FP32 in their order; the residues are then added in a
// fixed order through distributed shared memory. What bounds it is the longest sum: a structure of 128 atoms has
// P = 2 and up to 1300 terms in a row. So the four warps form the terms of a stage of reflections side by side, two to a packed FP32
// operation, into shared memory, and then add them in order, a warp per component x, y, z, B: six instructions a term
// on the chain instead of 55. 512 cells of 8 to 128 atoms: one 256-thread CTA a structure, a thread a sum, 203 us; a
// warp a CTA forming its own terms 160 us; 123 us now. The sums are the same bits in each form (k_grad_atoms_few too).
constexpr int kAtomCluster = 4;
constexpr int kAtomWarps = 8;
constexpr int kAtomCtaSums = 64;  // four warps for each 32
constexpr int kAtomSums = kAtomCtaSums * kAtomCluster;
constexpr int kAtomChunkRefl = 1024;
constexpr int kAtomStage = 256;  // reflections staged at most (divides kAtomChunkRefl)
constexpr int kAtomTerms = 64;   // terms of a sum formed per stage at most

__global__ void __launch_bounds__(32 * kAtomWarps, 4) k_grad_atoms(const GradArgs a)
{
    pdl_enter();
    __shared__ float4 red[kAtomCtaSums];
    __shared__ int4 si[kAtomStage];              // h, k, l and U of the staged reflections
    __shared__ float4 sf[kAtomStage];            // h, k, l and s^2
    __shared__ float sv[kAtomStage];             // V
    __shared__ float2 term[kAtomTerms][kAtomCtaSums];  // the two factors of each sum's terms
    const int ib = blockIdx.x / kAtomCluster, rank = blockIdx.x % kAtomCluster;  // the cluster is a row of the grid
    const int s = a.order[ib];
    const int64_t j0 = a.atom_off[s], j1 = a.atom_off[s + 1];
    const int w = (threadIdx.x >> 5) & 3, sum = (threadIdx.x & 31) + 32 * (threadIdx.x >> 7);  // this CTA's sum
    const int N = (int)(j1 - j0), t = kAtomCtaSums * rank + sum;
    const bool ok = !*a.abort_flag && a.geo[s].status == XRD_OK;  // the same for the whole cluster
    if (!ok) {
        if (j0 < 0 || j1 > a.n_atoms || N < 0) return;  // invalid atom offsets: touch nothing
        for (int i = rank * (int)blockDim.x + (int)threadIdx.x; i < N; i += kAtomCluster * blockDim.x) {
            a.d_frac[3 * (j0 + i)] = a.d_frac[3 * (j0 + i) + 1] = a.d_frac[3 * (j0 + i) + 2] = 0.f;
            a.d_B[j0 + i] = 0.f;
        }
        return;
    }
    const int64_t rb = a.refl_off[s];
    const int nr = (int)(a.refl_off[s + 1] - rb);
    const int Nc = min(N, kAtomSums);
    if (Nc == 0) return;
    const int P = kAtomSums / Nc;
    const int rho = t / Nc, al = t % Nc;
    const int stage = P >= 4 ? kAtomStage : (P >= 2 ? 2 : 1) * kAtomTerms;  // at most kAtomTerms terms a sum; divides kAtomChunkRefl
    const float2 k2 = make_float2(1.4629180792671596e-09f, 1.4629180792671596e-09f);
    for (int ac0 = 0; ac0 < N; ac0 += Nc) {
        const int at_i = ac0 + al;
        const bool valid = rho < P && at_i < N;
        float g = 0.f;  // component w of the sum
        Atom32 at{};
        Coef32 c{};
        if (valid) {
            at = a.atom32[j0 + at_i];
            c = a.coef32[at.z];
        }
        const float2 nb = make_float2(at.nb, at.nb), lo = make_float2(at.lo, at.lo), zf = make_float2(at.zf, at.zf);
        for (int r0 = 0; r0 < nr; r0 += kAtomChunkRefl) {
            const int hi = min(r0 + kAtomChunkRefl, nr);
            int i = r0 + rho;  // the sum's next reflection
            for (int b0 = r0; b0 < hi; b0 += stage) {
                const int be = min(b0 + stage, hi);
                __syncthreads();  // the previous stage's terms are added
                if ((int)threadIdx.x < be - b0) {
                    const int64_t r = rb + b0 + threadIdx.x;
                    const uint32_t key = a.key[r];
                    const int h = hkl_h(key), k = hkl_k(key), l = hkl_l(key);
                    si[threadIdx.x] = make_int4(h, k, l, __float_as_int(a.U[r]));
                    sf[threadIdx.x] = make_float4((float)h, (float)k, (float)l, d2f_pos(a.q[r]) * 0.25f);
                    sv[threadIdx.x] = a.V[r];
                }
                __syncthreads();
                const int m = valid && i < be ? (be - i + P - 1) / P : 0;  // the sum's terms in this stage
                for (int k0 = 2 * w; k0 < m; k0 += 8) {
                    const int i0 = i - b0 + k0 * P, i1 = k0 + 1 < m ? i0 + P : i0;
                    const int4 A0 = si[i0], A1 = si[i1];
                    const float2 s2 = make_float2(sf[i0].w, sf[i1].w);
                    const float2 U = make_float2(__int_as_float(A0.w), __int_as_float(A1.w)), V = make_float2(sv[i0], sv[i1]);
                    const uint32_t P0 = (uint32_t)A0.x * at.X + (uint32_t)A0.y * at.Y + (uint32_t)A0.z * at.Z;
                    const uint32_t P1 = (uint32_t)A1.x * at.X + (uint32_t)A1.y * at.Y + (uint32_t)A1.z * at.Z;
                    const float2 ph = __fmul2_rn(make_float2((float)(int32_t)P0, (float)(int32_t)P1), k2);
                    float2 sn, cs, e[4];
                    __sincosf(ph.x, &sn.x, &cs.x);
                    __sincosf(ph.y, &sn.y, &cs.y);
#pragma unroll
                    for (int j = 0; j < 4; j++) {
                        const float2 x = __fmul2_rn(make_float2(c.bl[j], c.bl[j]), s2);
                        e[j] = make_float2(ex2_approx(x.x), ex2_approx(x.y));
                    }
                    float2 f = __fmul2_rn(make_float2(c.a[3], c.a[3]), e[3]);
#pragma unroll
                    for (int j = 2; j >= 0; j--) f = __ffma2_rn(make_float2(c.a[j], c.a[j]), e[j], f);
                    f = __ffma2_rn(s2, f, zf);
                    const float2 x = __ffma2_rn(nb, s2, lo);
                    const float2 wt = __fmul2_rn(f, make_float2(ex2_approx(x.x), ex2_approx(x.y)));
                    const float2 us = __fmul2_rn(make_float2(-U.x, -U.y), sn);
                    const float2 t1 = __fmul2_rn(wt, __ffma2_rn(V, cs, us));
                    const float2 t2 = __fmul2_rn(wt, __ffma2_rn(U, cs, __fmul2_rn(V, sn)));
                    term[k0][sum] = make_float2(t1.x, t2.x);
                    if (k0 + 1 < m) term[k0 + 1][sum] = make_float2(t1.y, t2.y);
                }
                __syncthreads();
                const float* const coef = (const float*)sf + 4 * (i - b0) + w;
                const float* const tt = &term[0][sum].x + (w == 3 ? 1 : 0);
#pragma unroll 4
                for (int k = 0; k < m; k++) g = fmaf(coef[4 * k * P], tt[2 * kAtomCtaSums * k], g);
                i += m * P;
            }
        }
        ((float*)&red[sum])[w] = g;
        cluster_sync();  // every thread's sums stand
        if (w == 0 && rho == 0 && at_i < N) {
            float sx = 0.f, sy = 0.f, sz = 0.f, sb = 0.f;
            for (int p = 0; p < P; p++) {
                const int u = p * Nc + al;
                const float4 v = cluster_load(&red[u % kAtomCtaSums], u / kAtomCtaSums);
                sx += v.x;
                sy += v.y;
                sz += v.z;
                sb += v.w;
            }
            const int64_t o = j0 + a.atom32[j0 + at_i].src;
            const float fourpi = (float)(4.0 * kPi);
            a.d_frac[3 * o] = fourpi * sx;
            a.d_frac[3 * o + 1] = fourpi * sy;
            a.d_frac[3 * o + 2] = fourpi * sz;
            a.d_B[o] = -2.f * sb;
        }
        cluster_sync();  // read before the next chunk, or the exit, takes them away
    }
}

// The same sums for batches of few atoms a structure (kAtomFew on average): one CTA per structure, a thread a sum, which
// forms its own terms. With few atoms a structure's 256 sums are of few terms each, and what a cluster shares (staging by
// every CTA, three barriers a stage, the exchange) outweighs the shorter sums: a step of 3000 cells of 8 atoms on 1000
// points 556 us with clusters and 442 here, of one atom 1026 and 710, 50 000 cells of 4 atoms 4.65 and 2.91 ms; at 16
// cells of 8 atoms, or one, equal; 512 cells of 8 to 128 atoms 311 us with clusters and 411 here, 5000 cells of 27 atoms on
// average and up to 500 1.33 and 1.57 ms.
constexpr int kAtomFew = 8;

__global__ void __launch_bounds__(kAtomSums) k_grad_atoms_few(const GradArgs a)
{
    pdl_enter();
    __shared__ uint32_t skey[kAtomChunkRefl];
    __shared__ float ss2[kAtomChunkRefl], sU[kAtomChunkRefl], sV[kAtomChunkRefl];
    __shared__ float4 red[kAtomSums];
    const int s = a.order[blockIdx.x], t = threadIdx.x;
    const int64_t j0 = a.atom_off[s], j1 = a.atom_off[s + 1];
    const int N = (int)(j1 - j0);
    const bool ok = !*a.abort_flag && a.geo[s].status == XRD_OK;
    if (!ok) {
        if (j0 < 0 || j1 > a.n_atoms || N < 0) return;  // invalid atom offsets: touch nothing
        for (int i = t; i < N; i += kAtomSums) {
            a.d_frac[3 * (j0 + i)] = a.d_frac[3 * (j0 + i) + 1] = a.d_frac[3 * (j0 + i) + 2] = 0.f;
            a.d_B[j0 + i] = 0.f;
        }
        return;
    }
    const int64_t rb = a.refl_off[s];
    const int nr = (int)(a.refl_off[s + 1] - rb);
    const int Nc = min(N, kAtomSums);
    if (Nc == 0) return;
    const int P = kAtomSums / Nc, Pn = min(P, nr);
    const int rho = t / Nc, al = t % Nc;
    for (int ac0 = 0; ac0 < N; ac0 += Nc) {
        const int at_i = ac0 + al;
        const bool valid = rho < P && at_i < N;
        Atom32 at{};
        Coef32 c{};
        if (valid) {
            at = a.atom32[j0 + at_i];
            c = a.coef32[at.z];
        }
        float4 g = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int r0 = 0; r0 < nr; r0 += kAtomChunkRefl) {
            const int nc = min(kAtomChunkRefl, nr - r0);
            __syncthreads();
            for (int i = t; i < nc; i += kAtomSums) {
                skey[i] = a.key[rb + r0 + i];
                ss2[i] = d2f_pos(a.q[rb + r0 + i]) * 0.25f;
                sU[i] = a.U[rb + r0 + i];
                sV[i] = a.V[rb + r0 + i];
            }
            __syncthreads();
            for (int i = valid ? rho : nc; i < nc; i += P) {
                const uint32_t key = skey[i];
                const int h = hkl_h(key), k = hkl_k(key), l = hkl_l(key);
                const uint32_t Ph = (uint32_t)h * at.X + (uint32_t)k * at.Y + (uint32_t)l * at.Z;
                float sn, cs;
                __sincosf((float)(int32_t)Ph * 1.4629180792671596e-09f, &sn, &cs);
                const float s2 = ss2[i], U = sU[i], V = sV[i];
                const float e0 = ex2_approx(c.bl[0] * s2), e1 = ex2_approx(c.bl[1] * s2);
                const float e2 = ex2_approx(c.bl[2] * s2), e3 = ex2_approx(c.bl[3] * s2);
                const float f = fmaf(s2, fmaf(c.a[0], e0, fmaf(c.a[1], e1, fmaf(c.a[2], e2, c.a[3] * e3))), at.zf);
                const float wt = f * ex2_approx(fmaf(at.nb, s2, at.lo));
                const float t1 = wt * fmaf(V, cs, -U * sn), t2 = wt * fmaf(U, cs, V * sn);
                g.x = fmaf((float)h, t1, g.x);
                g.y = fmaf((float)k, t1, g.y);
                g.z = fmaf((float)l, t1, g.z);
                g.w = fmaf(s2, t2, g.w);
            }
        }
        red[t] = g;
        __syncthreads();
        if (rho == 0 && at_i < N) {
            float sx = 0.f, sy = 0.f, sz = 0.f, sb = 0.f;
            for (int p = 0; p < Pn; p++) {
                const float4 v = red[p * Nc + al];
                sx += v.x;
                sy += v.y;
                sz += v.z;
                sb += v.w;
            }
            const int64_t o = j0 + at.src;
            const float fourpi = (float)(4.0 * kPi);
            a.d_frac[3 * o] = fourpi * sx;
            a.d_frac[3 * o + 1] = fourpi * sy;
            a.d_frac[3 * o + 2] = fourpi * sz;
            a.d_B[o] = -2.f * sb;
        }
        __syncthreads();
    }
}

size_t broaden_smem_bytes(int n_pts, int W) { return sizeof(int) * (size_t)(n_pts + 2 * W + 3); }

void launch_broaden(const GradArgs& a, cudaStream_t st)
{
    if (a.n_struct <= 0) return;
    const size_t smem = broaden_smem_bytes(a.n_pts, a.W);
    if (smem > 48 * 1024) cudaFuncSetAttribute(k_broaden, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    launch_pdl(k_broaden, a.n_struct, a.n_struct <= kBroadenFew * a.sms ? kBroadenMaxThreads : kBroadenMaxThreads / 2, smem, st, a);
}

template <typename K>
static void launch_clusters(K k, const GradArgs& a, int cluster, int threads, bool pdl, cudaStream_t st)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)a.n_struct * cluster);
    cfg.blockDim = dim3(threads);
    cfg.stream = st;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cluster;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = pdl ? 2 : 1;
    cudaLaunchKernelEx(&cfg, k, a);
}

void launch_grad(const GradArgs& a, cudaStream_t st)
{
    if (a.n_struct <= 0) return;
    launch_clusters(k_grad_refl, a, kReflCluster, kReflThreads, false, st);
    if (a.n_atoms <= (int64_t)kAtomFew * a.n_struct) launch_pdl(k_grad_atoms_few, a.n_struct, kAtomSums, 0, st, a);
    else launch_clusters(k_grad_atoms, a, kAtomCluster, 32 * kAtomWarps, true, st);
}

}  // namespace xrd
