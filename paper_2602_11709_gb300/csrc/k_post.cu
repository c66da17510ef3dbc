// Steps S4-S6: sort by 2-theta, merge within the tolerance, hkl families,
// intensity cutoff and scaling, then compaction into dense CSR outputs.
//
// Sec. 2: reflections closer in 2-theta than a tolerance are merged into one
// peak, and the equivalent reflections of a peak are grouped into hkl families;
// the optional cutoff (Sec. 2) keeps peaks above
// a fraction of the largest one and Sec. 3 compares intensities on a 0-100 scale.
//
// One CTA per structure of up to 6144 reflections, held in shared memory (the
// larger ones run as the flat passes of k_post_flat.cu). The sort is a bucket
// sort in |g|^3 (reflections are uniform in the volume of the sphere, so
// buckets are nearly equally full); each reflection then takes its rank among
// the members of its own bucket on the full key (|g|^2, then -h, -k, -l), one
// thread per reflection.
// The anchor rule is sequential, so it is split: a reflection whose gap to its
// predecessor is >= tol always opens a peak (a definite start); the short runs
// between definite starts are resolved one thread per run.
#include <atomic>
#include <type_traits>

#include "xrd_internal.cuh"
#include "xrd_launch.h"
#include "xrd_post.cuh"

namespace xrd {

__host__ __device__ constexpr size_t align16(size_t x) { return (x + 15) & ~size_t(15); }

__host__ __device__ constexpr size_t post_smem_of(size_t c)
{
    // q, key, perm (16 bit), bucket ends, flags, peak starts, peak sums, family counts
    return align16(c * 8) + align16(c * 4) + align16(c * 2) + align16((c + 1) * 4) + align16(c) + align16(c * 4) +
           align16(c * 8) + align16(c * 4);
}

size_t post_smem_bytes(int cap) { return post_smem_of((size_t)cap); }

// The shared memory of a structure of up to CAP reflections
struct PostMem {
    double* q;
    uint32_t* key;
    uint16_t* perm;
    int* bkt;
    uint8_t* flag;
    int* pst;
    double* psum;
    int* fcnt;
    float* I;  // the FP32 variants' intensities, in the second half of psum
};
template <int CAP>
__device__ __forceinline__ PostMem post_mem()
{
    extern __shared__ __align__(16) unsigned char smem[];
    const size_t c = (size_t)CAP;
    PostMem m;
    unsigned char* p = smem;
    m.q = (double*)p; p += align16(c * 8);
    m.key = (uint32_t*)p; p += align16(c * 4);
    m.perm = (uint16_t*)p; p += align16(c * 2);
    m.bkt = (int*)p; p += align16((c + 1) * 4);
    m.flag = (uint8_t*)p; p += align16(c);
    m.pst = (int*)p; p += align16(c * 4);
    m.psum = (double*)p; p += align16(c * 8);
    m.fcnt = (int*)p;
    m.I = (float*)m.psum + c;
    return m;
}

// CTAs per SM that the shared memory of a class allows (228 KB per SM; about
// 2 KB more per CTA for the static arrays and the per-CTA reservation), at most
// 1024 threads: the launch bounds ask the compiler to fit that many CTAs in the
// register file too, and 64 registers a thread spill nothing. More threads gain nothing on large batches (100 000
// mixed cells 6.89 ms, 6.87 with 1280 threads, 6.89 with 1536) and their spills cost on small ones (256 hexagonal/P1
// cells 119, 124 and 133 us; 1024 small cells 190, 196 and 199 us).
__host__ __device__ constexpr int post_min_blocks(int cap, int nt)
{
    const int b = (int)((228u * 1024u) / (post_smem_of((size_t)cap) + 2048u));
    return b < 1 ? 1 : b * nt > 1024 ? 1024 / nt : b;
}

static __device__ TTab g_ttab[kTabN + 1];

__global__ void k_ttab_init()
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j > kTabN) return;
    const double th = (j * (double)kTabStepDeg) * (kPi / 360.0);
    const double sn = sin(th);
    const double S = sn * sn;
    TTab t;
    t.Sh = (float)S;
    t.Sl = (float)(S - (double)t.Sh);
    t.A = (float)sin(2.0 * th);
    t.Bc = (float)cos(2.0 * th);
    g_ttab[j] = t;
}

const TTab* init_tables(cudaStream_t st)
{
    k_ttab_init<<<(kTabN + 1 + 255) / 256, 256, 0, st>>>();
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_ttab) != cudaSuccess) return nullptr;
    return (const TTab*)p;
}

// The largest of all threads' values (bit patterns of floats >= 0), by one barrier; tmp: 32 words of shared memory,
// free after the caller's next barrier.
template <bool FI>
__device__ __forceinline__ unsigned long long post_max(unsigned long long v, unsigned long long* tmp)
{
    const int nw = blockDim.x >> 5, lane = threadIdx.x & 31;
    auto warp_max = [](unsigned long long x) -> unsigned long long {
        if constexpr (FI) {
            return __reduce_max_sync(0xffffffffu, (unsigned)x);
        } else {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) x = max(x, (unsigned long long)__shfl_xor_sync(0xffffffffu, x, o));
            return x;
        }
    };
    v = warp_max(v);
    if (lane == 0) tmp[threadIdx.x >> 5] = v;
    __syncthreads();
    return warp_max(lane < nw ? tmp[lane] : 0ull);
}

// The common case of a structure whose sorted reflections are all farther apart
// than the tolerance: every reflection is a peak of one family (g and -g, so
// multiplicity 2), and the merge runs, the peak-start scan and the family
// search are skipped. Same arithmetic and outputs as the general path.
template <typename PermT, bool FI>
__device__ void post_singles(const PostArgs& a, int s, int64_t base, int n, const double* q, const uint32_t* key,
                             const float* Is, const PermT* perm, uint8_t* flag, int* pst, double* psum, int* tmp,
                             double* dtmp)
{
    const int tid = threadIdx.x, nt = blockDim.x;
    double imax = 0.0, inv_imax = 0.0;
    float imaxf = 0.f, inv_imaxf = 0.f;
    unsigned long long lmax = 0;
    for (int p = tid; p < n; p += nt) {
        if (FI) {
            const float v = 2.f * Is[perm[p]];
            ((float*)psum)[p] = v;
            lmax = max(lmax, (unsigned long long)__float_as_uint(v));
        } else {
            const double v = 0.0 + 2.0 * a.I[base + perm[p]];
            psum[p] = v;
            lmax = max(lmax, dbits(v));
        }
    }
    const unsigned long long m = post_max<FI>(lmax, (unsigned long long*)dtmp);
    if (FI) {
        imaxf = __uint_as_float((uint32_t)m);
        inv_imaxf = imaxf > 0.f ? 1.f / imaxf : 0.f;
    } else {
        imax = __longlong_as_double((long long)m);
        inv_imax = imax > 0.0 ? 1.0 / imax : 0.0;
    }
    const uint32_t thrf = __float_as_uint((float)a.cutoff * imaxf);
    const unsigned long long thr = dbits(a.cutoff * imax);
    auto keep = [&](int p) -> int {
        return a.cutoff == 0.0 || (FI ? __float_as_uint(((float*)psum)[p]) > thrf : dbits(psum[p]) > thr);
    };
    const int nk = block_scan_to(n, tmp, keep, [&](int p, int sum, int v) {
        flag[p] = v;
        pst[p] = sum;
    });
    __syncthreads();
    for (int p = tid; p < n; p += nt) {
        if (!flag[p]) continue;
        const int64_t o = base + pst[p];
        const int v = perm[p];
        a.st_q[o] = q[v];
        if (FI) {
            const float ps = ((const float*)psum)[p];
            ((float*)a.st_I)[o] = (a.scaled && imaxf > 0.f) ? (ps == imaxf ? 100.f : 100.f * (ps * inv_imaxf)) : ps;
        } else {
            const double ps = psum[p];
            a.st_I[o] = (a.scaled && imax > 0.0) ? (ps == imax ? 100.0 : 100.0 * (ps * inv_imax)) : ps;
        }
        a.st_foff[o] = pst[p];  // one family per kept peak
        const uint32_t rep = key[v];
        a.st_key[o] = rep;
        a.st_mult[o] = 2;
    }
    if (tid == 0) {
        a.npk[s] = nk;
        a.nfm[s] = nk;
    }
}

// Sum of a peak's intensities (each half-space reflection stands for g and -g): the same operations whoever sums.
__device__ __forceinline__ float peak_add(float sum, float v, bool first) { return first ? 2.f * v : fmaf(2.f, v, sum); }
__device__ __forceinline__ double peak_add(double sum, double v, bool first) { return (first ? 0.0 : sum) + 2.0 * v; }

// A peak of up to 32 C members at merge positions i0 .. i0 + m - 1, by a whole warp, C members to a lane: the members'
// intensities summed in merge order (every lane gets the sum), and the families found by one round of comparisons
// against each member in turn. A family leaves its representative (the largest packed key) and its size (from the
// second family on) in the key and |g|^2 slots of the peak's member of its rank, by descending representative.
// Returns the number of families.
constexpr int kWarpPeak = 128;
template <int C, typename PermT, bool FI, typename FK, typename T>
__device__ __forceinline__ int merged_peak_body(FK fk, double* q, uint32_t* key, const PermT* perm, int i0, int m,
                                                const float* Is, const double* I, T& sum)
{
    const int lane = threadIdx.x & 31;
    int v[C], cnt[C], rank[C];
    T Iv[C];
    unsigned long long k[C];
    uint32_t kv[C], rep[C];
    bool lead[C];
#pragma unroll
    for (int c = 0; c < C; c++) {
        const int i = 32 * c + lane, at = i0 + (i < m ? i : 0);
        v[c] = perm[at];
        if constexpr (FI) Iv[c] = Is[v[c]];
        else Iv[c] = I[v[c]];
        k[c] = fk(at);
        kv[c] = key[v[c]];
        lead[c] = i < m;
        cnt[c] = 0;
        rank[c] = 0;
        rep[c] = 0;
    }
    sum = (T)0;
#pragma unroll
    for (int b = 0; b < C; b++) {
        const int mb = min(32, m - 32 * b);
        for (int j = 0; j < mb; j++) {
            sum = peak_add(sum, __shfl_sync(0xffffffffu, Iv[b], j), b == 0 && j == 0);
            const unsigned long long kj = __shfl_sync(0xffffffffu, k[b], j);
            const uint32_t kvj = __shfl_sync(0xffffffffu, kv[b], j);
#pragma unroll
            for (int c = 0; c < C; c++)
                if (kj == k[c]) {
                    cnt[c]++;
                    rep[c] = max(rep[c], kvj);
                    lead[c] = lead[c] && 32 * b + j >= 32 * c + lane;
                }
        }
    }
    unsigned leaders[C];
    int nf = 0;
#pragma unroll
    for (int b = 0; b < C; b++) {
        leaders[b] = __ballot_sync(0xffffffffu, lead[b]);
        nf += __popc(leaders[b]);
        for (unsigned u = leaders[b]; u; u &= u - 1) {
            const uint32_t r = __shfl_sync(0xffffffffu, rep[b], __ffs(u) - 1);
#pragma unroll
            for (int c = 0; c < C; c++) rank[c] += r > rep[c];
        }
    }
    __syncwarp();  // every key is read
#pragma unroll
    for (int c = 0; c < C; c++)
        if (lead[c]) {
            const int slot = perm[i0 + rank[c]];
            key[slot] = rep[c];
            if (rank[c] > 0) q[slot] = __longlong_as_double(cnt[c]);
        }
    return nf;
}
// out of line: few peaks have more than 32 members
template <typename PermT, bool FI, typename FK, typename T>
__device__ __noinline__ int merged_peak_large(FK fk, double* q, uint32_t* key, const PermT* perm, int i0, int m,
                                              const float* Is, const double* I, T& sum)
{
    return merged_peak_body<kWarpPeak / 32, PermT, FI>(fk, q, key, perm, i0, m, Is, I, sum);
}

template <typename PermT>
struct FamilyKeys {  // family key of the member at merge position i
    const unsigned long long* fkg;
    const uint32_t* key;
    const PermT* perm;
    bool hex;
    __device__ __forceinline__ unsigned long long operator()(int i) const
    {
        return fkg ? fkg[perm[i]] : family_key(key[perm[i]], hex);
    }
};
// The same for a peak of any number of members (rare, by tolerances far above a line's width): each member's
// representative (0 unless it is the first of its family) and family size go through trep and tcnt, m words each of the
// structure's output staging, which is free until the peaks are done. A thread each, which compares every member with
// every family of the peak and again for the ranks, took 4.4 s on 30 small cells at a tolerance of 5 degrees; now 1 ms.
template <typename PermT, bool FI, typename T>
__device__ __forceinline__ int merged_peak_any(FamilyKeys<PermT> fk, double* q, uint32_t* key, const PermT* perm, int i0, int m,
                                            const float* Is, const double* I, uint32_t* trep, int* tcnt, T& sum)
{
    constexpr int C = kWarpPeak / 32;
    const int lane = threadIdx.x & 31;
    sum = (T)0;
    for (int j0 = 0; j0 < m; j0 += 32) {
        const int v = perm[i0 + min(j0 + lane, m - 1)];
        T Iv;
        if constexpr (FI) Iv = Is[v];
        else Iv = I[v];
        for (int j = 0; j < min(32, m - j0); j++) sum = peak_add(sum, __shfl_sync(0xffffffffu, Iv, j), j0 + j == 0);
    }
    int nf = 0;
    for (int b0 = 0; b0 < m; b0 += 32 * C) {
        unsigned long long k[C];
        uint32_t rep[C];
        int cnt[C];
        bool lead[C];
#pragma unroll
        for (int c = 0; c < C; c++) {
            const int i = b0 + 32 * c + lane;
            k[c] = fk(i0 + min(i, m - 1));
            rep[c] = 0;
            cnt[c] = 0;
            lead[c] = i < m;
        }
        for (int j0 = 0; j0 < m; j0 += 32) {
            const int at = i0 + min(j0 + lane, m - 1);
            const unsigned long long kl = fk(at);
            const uint32_t kvl = key[perm[at]];
            for (int j = 0; j < min(32, m - j0); j++) {
                const unsigned long long kj = __shfl_sync(0xffffffffu, kl, j);
                const uint32_t kvj = __shfl_sync(0xffffffffu, kvl, j);
#pragma unroll
                for (int c = 0; c < C; c++)
                    if (kj == k[c]) {
                        cnt[c]++;
                        rep[c] = max(rep[c], kvj);
                        lead[c] = lead[c] && j0 + j >= b0 + 32 * c + lane;
                    }
            }
        }
#pragma unroll
        for (int c = 0; c < C; c++) {
            const int i = b0 + 32 * c + lane;
            if (i < m) {
                trep[i] = lead[c] ? rep[c] : 0u;
                tcnt[i] = cnt[c];
            }
            nf += __popc(__ballot_sync(0xffffffffu, lead[c]));
        }
    }
    __syncwarp();  // every key is read, trep and tcnt are written
    for (int b0 = 0; b0 < m; b0 += 32) {
        const int i = b0 + lane;
        const uint32_t r = i < m ? trep[i] : 0u;
        int rank = 0;
        if (!__ballot_sync(0xffffffffu, r != 0u)) continue;
        for (int j0 = 0; j0 < m; j0 += 32) {
            const uint32_t rl = j0 + lane < m ? trep[j0 + lane] : 0u;
            for (int j = 0; j < 32; j++) rank += __shfl_sync(0xffffffffu, rl, j) > r;
        }
        if (r != 0u) {
            const int slot = perm[i0 + rank];
            key[slot] = r;
            if (rank > 0) q[slot] = __longlong_as_double(tcnt[i]);
        }
    }
    return nf;
}
// all of them, listed at the end of m.pst (n: the structure's reflections)
template <int CAP, bool FI>
__device__ __noinline__ void merged_peaks_any(const PostArgs& a, int64_t base, bool hex, int n, int nlist)
{
    using T = typename std::conditional<FI, float, double>::type;
    const PostMem m = post_mem<CAP>();
    const FamilyKeys<uint16_t> fk{a.fkg ? a.fkg + base : nullptr, m.key, m.perm, hex};
    for (int li = threadIdx.x >> 5; li < nlist; li += blockDim.x >> 5) {
        const int p = m.pst[n - 1 - li], i0 = m.bkt[p], mp = m.bkt[p + 1] - i0;
        T sum;
        const int nf = merged_peak_any<uint16_t, FI>(fk, m.q, m.key, m.perm, i0, mp, m.I, FI ? nullptr : a.I + base,
                                                     a.st_key + base + i0, a.st_mult + base + i0, sum);
        if ((threadIdx.x & 31) == 0) {
            ((T*)m.psum)[p] = sum;
            m.fcnt[p] = nf;
        }
    }
}

// FI: intensities are FP32 (the FP32 structure-factor variants) and peak sums,
// cutoff and scaling run in FP32; otherwise FP64 throughout.
// hex: Miller-Bravais families. ahead(0), ahead(1): called once each by all threads, in this order, where the work in
// between hides the latency of a global load.
// The phases are short (a few elements a thread), so barriers and the latency of passes through shared memory bound
// them: loading and counting are one pass, the flags are the peak starts, the peak list, the cutoff and the offsets come
// out of the scans themselves, and the next structure is claimed meanwhile (16 barriers a structure; with a pass for
// each of these, 25 barriers and the claim in the open, 100 000 mixed cells took 7.06 ms a call, now 6.89; 20 000 at
// Mo K-alpha 6.31, now 6.17).
template <int CAP, typename PermT, bool FI, typename Ahead>
__device__ void post_structure(const PostArgs& a, int s, int64_t base, int n, bool hex, double* q, uint32_t* key,
                               float* Is, PermT* perm, int* bkt, uint8_t* flag, int* pst, double* psum, int* fcnt,
                               int* tmp, double* dtmp, Ahead ahead)
{
    const int tid = threadIdx.x, nt = blockDim.x;
    const float l2 = a.l2f, lh = a.lhf, ttol = a.ttol;
    const double lam = a.lambda, tol = a.tol;
    // family key of the member at merge position i: the caller's point group (precomputed per
    // reflection), else permutation and sign (Miller-Bravais for a hexagonal cell)
    const FamilyKeys<PermT> fk{a.fkg ? a.fkg + base : nullptr, key, perm, hex};
    // ---- bucket sort on |g|^3 in [r2min^1.5, r2max^1.5] (a monotone map of |g|^2) ----
    // fcnt holds each reflection's bucket and pst the bucket-ordered reflections
    // until the merge step needs them.
    int* const bid = fcnt;
    int* const perm1 = pst;
    const int nb = n;
    const float lo3 = a.lo3, hi3 = a.hi3;
    const float scale = (float)nb / (hi3 - lo3);
    for (int i = tid; i <= nb; i += nt) bkt[i] = 0;
    __syncthreads();
    for (int i = tid; i < n; i += nt) {
        const double qi = a.q[base + i];
        q[i] = qi;
        key[i] = a.key[base + i];
        if (FI) Is[i] = a.If[base + i];
        const float qf = d2f_pos(qi);
        int b = (int)((qf * sqrtf(qf) - lo3) * scale);
        b = min(max(b, 0), nb - 1);
        bid[i] = b;
        atomicAdd(&bkt[b], 1);
    }
    __syncthreads();
    block_excl_scan(bkt, nb, tmp);
    ahead(0);
    for (int i = tid; i < n; i += nt) perm1[atomicAdd(&bkt[bid[i]], 1)] = i;
    __syncthreads();
    // bkt[b] is now the end of bucket b; rank within the bucket gives the position
    for (int p = tid; p < n; p += nt) {
        const int v = perm1[p];
        const int b = bid[v];
        const int b0 = b ? bkt[b - 1] : 0, b1 = bkt[b];
        int r = b0;
        if (b1 - b0 > 1) {
            const double qv = q[v];
            const uint32_t kv = key[v];
            for (int j = b0; j < b1; j++) {
                const int u = perm1[j];
                r += before(q[u], key[u], qv, kv);  // false for u == v
            }
        }
        perm[r] = (PermT)v;
    }
    __syncthreads();
    // ---- the caller's per-reflection list, in merge order ----
    if (a.refl_hkl && base + n <= a.cap_refl) {
        for (int p = tid; p < n; p += nt) {
            const int v = perm[p];
            const int64_t o = base + p;
            const uint32_t kv = key[v];
            a.refl_hkl[3 * o] = hkl_h(kv);
            a.refl_hkl[3 * o + 1] = hkl_k(kv);
            a.refl_hkl[3 * o + 2] = hkl_l(kv);
            float qh, ql;
            split_pos(q[v], qh, ql);
            a.refl_tt[o] = two_theta_out(qh, ql, a.l2h, a.l2l, a.ttab);
            a.refl_I[o] = FI ? (double)Is[v] : a.I[base + v];
        }
    }
    // ---- anchor merge: definite starts, then one thread per run ----
    int close_pair = 0;
    for (int i = tid; i < n; i += nt) {
        const bool start = (i == 0) || !tt_close(q[perm[i - 1]], q[perm[i]], l2, lh, ttol, lam, tol);
        flag[i] = start;
        pst[i] = start;
        close_pair |= !start;
    }
    ahead(1);
    if (!__syncthreads_or(close_pair)) {  // no two reflections within the tolerance: every one is a peak
        post_singles<PermT, FI>(a, s, base, n, q, key, Is, perm, flag, pst, psum, tmp, dtmp);
        return;
    }
    for (int i = tid; i < n; i += nt) {
        if (!flag[i] || i + 1 >= n || flag[i + 1]) continue;
        double qa = q[perm[i]];
        int e = i + 2;  // end of the run: the next definite start, four flags at a time where they are aligned
        while (e < n && !flag[e]) e += (e & 3) == 0 && e + 4 <= n && *(const uint32_t*)(flag + e) == 0u ? 4 : 1;
        // |g|^2 ascends, so a last member within the tolerance of the first one has all others within it too
        if (tt_close(qa, q[perm[e - 1]], l2, lh, ttol, lam, tol)) continue;
        for (int j = i + 1; j < e; j++) {
            const double qj = q[perm[j]];
            if (!tt_close(qa, qj, l2, lh, ttol, lam, tol)) {
                pst[j] = 1;
                qa = qj;
            }
        }
    }
    __syncthreads();
    // bkt becomes the list of peak start positions
    const int np = block_scan_to(n, tmp, [&](int i) { return pst[i]; }, [&](int i, int id, int start) {
        if (start) bkt[id] = i;
    });
    if (tid == 0) {
        bkt[np] = n;
        bkt[np + 1] = 0;  // merged peaks of more than one member (np < n here)
    }
    __syncthreads();
    // ---- per peak: merged intensity (each half-space reflection stands for g and -g) and families ----
    // A peak of one member is its thread's; one of more goes to a list (pst is free until the cutoff)
    // that the warps work off (merged_peak). One thread a peak took most of the structure's time where peaks have many
    // members: rock salt (293 reflections, peaks of up to 36) 62 000 of 105 000 cycles, and 13 000 more in the staging.
    // Peak sums are >= 0, so their maximum is taken through the bit patterns.
    using T = typename std::conditional<FI, float, double>::type;
    T* const ps = (T*)psum;
    auto member_I = [&](int v) -> T {
        if constexpr (FI) return Is[v];
        else return a.I[base + v];
    };
    auto bits_of = [](T v) -> unsigned long long {
        if constexpr (FI) return __float_as_uint(v);
        else return dbits(v);
    };
    unsigned long long lmax = 0;
    for (int p = tid; p < np; p += nt) {
        const int i0 = bkt[p], m = bkt[p + 1] - i0;
        if (m > kWarpPeak) {  // from the list's end, counted in the upper half
            pst[n - 1 - (atomicAdd(&bkt[np + 1], 1 << 16) >> 16)] = p;
            continue;
        }
        if (m > 1) {
            pst[atomicAdd(&bkt[np + 1], 1) & 0xffff] = p;
            continue;
        }
        const T sum = peak_add((T)0, member_I(perm[i0]), true);
        ps[p] = sum;
        fcnt[p] = 1;
        lmax = max(lmax, bits_of(sum));
    }
    __syncthreads();
    const int nmulti = bkt[np + 1] & 0xffff, nlarge = bkt[np + 1] >> 16;
    const double* const Id = FI ? nullptr : a.I + base;
    for (int li = tid >> 5; li < nmulti; li += nt >> 5) {
        const int p = pst[li], i0 = bkt[p], m = bkt[p + 1] - i0;
        T sum;
        int nf;
        if (m <= 32) nf = merged_peak_body<1, PermT, FI>(fk, q, key, perm, i0, m, Is, Id, sum);
        else nf = merged_peak_large<PermT, FI>(fk, q, key, perm, i0, m, Is, Id, sum);
        if ((tid & 31) == 0) {
            ps[p] = sum;
            fcnt[p] = nf;
            lmax = max(lmax, bits_of(sum));
        }
    }
    if (nlarge) {
        merged_peaks_any<CAP, FI>(a, base, hex, n, nlarge);
        __syncthreads();
        for (int li = tid; li < nlarge; li += nt) lmax = max(lmax, bits_of(ps[pst[n - 1 - li]]));
    }
    const unsigned long long mbits = post_max<FI>(lmax, (unsigned long long*)dtmp);
    T imax, inv_imax;
    unsigned long long thr;
    if constexpr (FI) {
        imax = __uint_as_float((uint32_t)mbits);
        inv_imax = imax > 0.f ? 1.f / imax : 0.f;
        thr = __float_as_uint((float)a.cutoff * imax);
    } else {
        imax = __longlong_as_double((long long)mbits);
        thr = dbits(a.cutoff * imax);
        if (tid == 0) dtmp[32] = imax > 0.0 ? 1.0 / imax : 0.0;
        __syncthreads();
        inv_imax = dtmp[32];
    }
    // ---- cutoff and the offsets of kept peaks (upper half) and their families (at most 6144 each) ----
    const int kf = block_scan_to(
        np, tmp, [&](int p) { return a.cutoff == 0.0 || bits_of(ps[p]) > thr ? 1 << 16 | fcnt[p] : 0; },
        [&](int p, int sum, int v) {
            flag[p] = v != 0;
            pst[p] = sum;
        });
    const int nk = kf >> 16, nf = kf & 0xffff;
    __syncthreads();
    for (int p = tid; p < np; p += nt) {
        if (!flag[p]) continue;
        const int i0 = bkt[p], m = bkt[p + 1] - i0, f0 = pst[p] & 0xffff;
        const int64_t o = base + (pst[p] >> 16);
        a.st_q[o] = q[perm[i0]];  // anchor |g|^2: 2-theta and d are formed during compaction
        const T v = ps[p];        // the largest peak maps to exactly 100
        ((T*)a.st_I)[o] = (a.scaled && imax > (T)0) ? (v == imax ? (T)100 : (T)100 * (v * inv_imax)) : v;
        a.st_foff[o] = f0;
        const int nfp = fcnt[p];
        int first = m;  // members of the first family: those of no other
        for (int r = nfp - 1; r >= 0; r--) {
            const int u = perm[i0 + r], c = r ? (int)__double_as_longlong(q[u]) : first;
            first -= c;
            a.st_key[base + f0 + r] = key[u];
            a.st_mult[base + f0 + r] = 2 * c;
        }
    }
    if (tid == 0) {
        a.npk[s] = nk;
        a.nfm[s] = nf;
    }
}

// An asynchronous copy of N bytes (4 or 8, aligned) to shared memory, and the wait for the thread's copies
template <int N>
__device__ __forceinline__ void copy_async(void* to, const void* from)
{
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;"
                 :: "r"((uint32_t)__cvta_generic_to_shared(to)), "l"(from), "n"(N) : "memory");
}
__device__ __forceinline__ void copy_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// A claimed structure: its extent in the reflection arrays, hexagonal, with an invalid atom
struct PostClaim {
    int64_t base, end;
    int s, hex, bad;
};

// Persistent CTAs over one size class of structures (a list built by the scan
// kernel, largest first), each CTA claiming the next structure from a counter
// while it works on the current one.
// The structure's reflections live in shared memory (n <= CAP); the FP32
// variants also stage the intensities there, in the second half of the
// peak-sum area (FP32 peak sums use the first half).
template <int CAP, int NT, bool FI>
__global__ void __launch_bounds__(NT, post_min_blocks(CAP, NT)) k_post(const PostArgs a, int c_lo, int c_hi, bool first)
{
    static_assert(CAP > 0, "the largest class runs as the flat passes");
    pdl_chain_enter(first);
    __shared__ int tmp[32];
    __shared__ double dtmp[33];
    __shared__ PostClaim claims[2];
    if (*a.abort_flag) {
        pdl_chain_exit();
        return;
    }
    // thread 0's claim of the next structure while the CTA works on the current one: the queue's counter, then the
    // structure from its class's list (step 0), then its extent (1), each copied to shared memory without waiting for it
    auto list = [&](int li, PostClaim& c) {
        int cls = c_hi;  // the larger classes first
        while (cls >= c_lo && li >= a.cls_cnt[cls]) li -= a.cls_cnt[cls--];
        if (cls >= c_lo) copy_async<4>(&c.s, a.cls_list + (int64_t)cls * a.n_struct + li);
        else c.s = -1;
    };
    auto extent = [&](PostClaim& c) {
        copy_async_wait();
        if (c.s < 0) return;
        copy_async<8>(&c.base, a.refl_off + c.s);
        copy_async<8>(&c.end, a.refl_off + c.s + 1);
        copy_async<4>(&c.hex, &a.geo[c.s].hex);
        if (a.atom_bad) copy_async<4>(&c.bad, a.atom_bad + c.s);
        else c.bad = 0;
    };
    if (threadIdx.x == 0) {
        list(atomicAdd(a.cls_next + c_lo, 1), claims[0]);
        extent(claims[0]);
        copy_async_wait();
    }
    for (int k = 0;; k ^= 1) {
        __syncthreads();  // the previous structure is done with shared memory, the claim is written
        const PostClaim cl = claims[k];
        const int s = cl.s;
        if (s < 0) break;
        const int64_t base = cl.base;
        const int n = (int)(cl.end - base);
        int li = 0;
        if (threadIdx.x == 0) li = atomicAdd(a.cls_next + c_lo, 1);
        auto ahead = [&](int step) {
            if (threadIdx.x) return;
            if (step == 0) list(li, claims[k ^ 1]);
            else extent(claims[k ^ 1]);
        };
        if (cl.bad || n == 0) {
            if (threadIdx.x == 0) {
                a.npk[s] = 0;
                a.nfm[s] = 0;
                if (cl.bad && a.status[s] == XRD_OK) {  // an invalid atom: no peaks, the structure reports XRD_EINVAL
                    a.status[s] = XRD_EINVAL;
                    atomicAdd((unsigned long long*)&a.totals[3], 1ull);
                }
            }
            ahead(0);
            ahead(1);
        } else {
            const PostMem m = post_mem<CAP>();
            post_structure<CAP, uint16_t, FI>(a, s, base, n, cl.hex != 0, m.q, m.key, m.I, m.perm, m.bkt, m.flag, m.pst,
                                              m.psum, m.fcnt, tmp, dtmp, ahead);
        }
        if (threadIdx.x == 0) copy_async_wait();
    }
    pdl_chain_exit();
}

// Exclusive scans of kept peaks and families per structure (single block),
// output capacity check, totals. The structures are walked in chunks of
// kOutItems * blockDim: coalesced loads into registers, then a transpose
// through shared memory so that each thread scans consecutive structures.
constexpr int kOutThreads = 1024;
constexpr int kOutItems = 4;

__global__ void __launch_bounds__(kOutThreads) k_scan_out(const CompactArgs a)
{
    pdl_enter();
    __shared__ long long ws[33];
    __shared__ long long buf[kOutItems * kOutThreads];
    if (*a.abort_flag) return;
    const int n = a.n_struct, nt = blockDim.x, tid = threadIdx.x, CH = kOutItems * nt;
    long long cp = 0, cf = 0;
    for (int base = 0; base < n; base += CH) {
        long long vp[kOutItems], vf[kOutItems];
#pragma unroll
        for (int u = 0; u < kOutItems; u++) {
            const int i = base + u * nt + tid;
            vp[u] = i < n ? a.npk[i] : 0;
            vf[u] = i < n ? a.nfm[i] : 0;
        }
        long long tp, tf;
        chunk_scan<kOutItems>(vp, buf, ws, &tp);
        chunk_scan<kOutItems>(vf, buf, ws, &tf);
#pragma unroll
        for (int u = 0; u < kOutItems; u++) {
            const int i = base + u * nt + tid;
            if (i < n) {
                a.out.peak_off[i] = cp + vp[u];
                a.fam_soff[i] = cf + vf[u];
                if (a.out.refl_off) a.out.refl_off[i] = a.refl_off[i];
            }
        }
        cp += tp;
        cf += tf;
    }
    const bool over = cp > a.cap_peaks || cf > a.cap_fam || (a.out.refl_off && a.refl_off[n] > a.out.cap_refl);
    if (over)
        for (int i = tid; i < n; i += nt) a.out.status[i] = XRD_ECAPACITY;
    if (tid == 0) {
        a.out.peak_off[n] = cp;
        a.fam_soff[n] = cf;
        a.out.totals[1] = cp;
        a.out.totals[2] = cf;
        if (a.out.refl_off) a.out.refl_off[n] = a.refl_off[n];
        *a.out_abort = over;
        if (over) a.out.totals[3] = n;
        else a.out.fam_off[cp] = cf;
    }
}

// Multi-block form of k_scan_out for batches of more than two chunks: chunk
// sums of kept peaks and families first, then every chunk scans its own
// structures from the sums of the chunks before it.
__global__ void __launch_bounds__(kOutThreads) k_scan_out_parts(const CompactArgs a)
{
    pdl_enter();
    __shared__ long long ws[33];
    if (*a.abort_flag) return;
    const int n = a.n_struct, nt = blockDim.x, tid = threadIdx.x, base = blockIdx.x * kOutItems * nt;
    long long p = 0, f = 0;
#pragma unroll
    for (int u = 0; u < kOutItems; u++) {
        const int i = base + u * nt + tid;
        if (i < n) {
            p += a.npk[i];
            f += a.nfm[i];
        }
    }
    long long tp, tf;
    block_prefix_ll(p, ws, &tp);
    block_prefix_ll(f, ws, &tf);
    if (tid == 0) {
        a.parts[2 * blockIdx.x] = tp;
        a.parts[2 * blockIdx.x + 1] = tf;
    }
}

__global__ void __launch_bounds__(kOutThreads) k_scan_out_final(const CompactArgs a)
{
    pdl_enter();
    __shared__ long long ws[33];
    __shared__ long long buf[kOutItems * kOutThreads];
    __shared__ long long pre[2], all[2];
    if (*a.abort_flag) return;
    const int n = a.n_struct, nt = blockDim.x, tid = threadIdx.x, b = blockIdx.x, base = b * kOutItems * nt;
    if (tid < 2) {
        long long q = 0, t = 0;
        for (int c = 0; c < (int)gridDim.x; c++) {
            const long long v = a.parts[2 * c + tid];
            q += c < b ? v : 0;
            t += v;
        }
        pre[tid] = q;
        all[tid] = t;
    }
    __syncthreads();
    const long long cp = all[0], cf = all[1];
    const bool over = cp > a.cap_peaks || cf > a.cap_fam || (a.out.refl_off && a.refl_off[n] > a.out.cap_refl);
    long long vp[kOutItems], vf[kOutItems], tp, tf;
#pragma unroll
    for (int u = 0; u < kOutItems; u++) {
        const int i = base + u * nt + tid;
        vp[u] = i < n ? a.npk[i] : 0;
        vf[u] = i < n ? a.nfm[i] : 0;
    }
    chunk_scan<kOutItems>(vp, buf, ws, &tp);
    chunk_scan<kOutItems>(vf, buf, ws, &tf);
#pragma unroll
    for (int u = 0; u < kOutItems; u++) {
        const int i = base + u * nt + tid;
        if (i < n) {
            a.out.peak_off[i] = pre[0] + vp[u];
            a.fam_soff[i] = pre[1] + vf[u];
            if (a.out.refl_off) a.out.refl_off[i] = a.refl_off[i];
            if (over) a.out.status[i] = XRD_ECAPACITY;
        }
    }
    if (b == 0 && tid == 0) {
        if (a.out.refl_off) a.out.refl_off[n] = a.refl_off[n];
        a.out.peak_off[n] = cp;
        a.fam_soff[n] = cf;
        a.out.totals[1] = cp;
        a.out.totals[2] = cf;
        *a.out_abort = over;
        if (over) a.out.totals[3] = n;
        else a.out.fam_off[cp] = cf;
    }
}

// largest s in [lo, n) with off[s] <= i, for off[lo] <= i < off[n]
__device__ __forceinline__ int owner(const int64_t* __restrict__ off, int lo, int n, int64_t i)
{
    int hi = n;
    while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (off[mid] <= i) lo = mid;
        else hi = mid;
    }
    return lo;
}

// Kept peaks and their families into the dense CSR outputs. Each warp takes one contiguous range of output peaks,
// finds its first structure by bisection and walks the structures forward: what belongs to a structure is read once
// per segment, its peaks and its families are each a contiguous range of the staging and of the outputs, and the
// three indices of a family leave as consecutive words (a shuffle transposes 32 packed keys). 2-theta and d are
// formed here from the anchor |g|^2. Bound by HBM and by what hides its latency: 54 M peaks of 100 000 mixed cells (3.9 GB) took
// 949 us with a thread per peak that looked up its structure and wrote its families one word in three (415
// instructions per 32 peaks), 732 us (270 instructions) now, 5.3 of the 6.8 TB/s that a copy reaches.
constexpr int kCompactThreads = 256;
constexpr int kCompactCtas = 4;   // CTAs per SM: one wave
constexpr int kCompactBatch = 4;  // peaks or families a lane has in flight

__global__ void __launch_bounds__(kCompactThreads, kCompactCtas) k_compact(const CompactArgs a)
{
    pdl_enter();
    if (*a.abort_flag || *a.out_abort) return;
    const int n = a.n_struct, lane = threadIdx.x & 31;
    const int64_t* __restrict__ poff = a.out.peak_off;
    const int64_t total = poff[n];
    int64_t warps = (int64_t)gridDim.x * (kCompactThreads / 32);
    int64_t w = (int64_t)blockIdx.x * (kCompactThreads / 32) + (threadIdx.x >> 5);
    // few outputs: half of the warps take the peaks and half the families, so that neither waits for the other
    const bool split = total <= 16 * warps, peaks = !split || !(w & 1), fams = !split || (w & 1);
    if (split) {
        warps >>= 1;
        w >>= 1;
    }
    const int64_t per = ((total + warps - 1) / warps + 31) & ~31ll;
    const int64_t start = w * per;
    const int64_t end = min(start + per, total);
    if (start >= end) return;
    const double* __restrict__ st_q = a.st_q;
    const float* __restrict__ st_If = (const float*)a.st_I;
    const int* __restrict__ st_foff = a.st_foff;
    const uint32_t* __restrict__ st_key = a.st_key;
    const int* __restrict__ st_mult = a.st_mult;
    double* __restrict__ o_tt = a.out.two_theta;
    double* __restrict__ o_d = a.out.d_hkl;
    double* __restrict__ o_I = a.out.intensity;
    int64_t* __restrict__ o_fo = a.out.fam_off;
    int32_t* __restrict__ o_hkl = a.out.hkl;
    int32_t* __restrict__ o_mult = a.out.mult;
    int s = owner(poff, 0, n, start);
    int64_t P = start, ps = poff[s], pe = poff[s + 1];
    while (P < end) {
        while (pe <= P) {  // the next structure with peaks
            s++;
            ps = pe;
            pe = poff[s + 1];
        }
        const int64_t rb = a.refl_off[s], fs = a.fam_soff[s];
        const int64_t stop = min(pe, end);
        const int64_t shift = rb - ps;  // staging index of output peak P: P + shift
        // the families of these peaks, as offsets within the structure
        const int f0 = st_foff[P + shift], f1 = stop < pe ? st_foff[stop + shift] : (int)(a.fam_soff[s + 1] - fs);
        for (int64_t p0 = peaks ? P : stop; p0 < stop; p0 += 32 * kCompactBatch) {  // loads of a batch before its stores
            double qa[kCompactBatch];
            int fo[kCompactBatch];
            float If[kCompactBatch];
#pragma unroll
            for (int u = 0; u < kCompactBatch; u++) {
                const int64_t p = min(p0 + 32 * u + lane, stop - 1) + shift;
                qa[u] = st_q[p];
                fo[u] = st_foff[p];
                If[u] = a.fi ? st_If[p] : 0.f;
            }
#pragma unroll
            for (int u = 0; u < kCompactBatch; u++) {
                const int64_t p = p0 + 32 * u + lane;
                if (p >= stop) break;
                float qh, ql;
                split_pos(qa[u], qh, ql);
                o_tt[p] = two_theta_out(qh, ql, a.l2h, a.l2l, a.ttab);
                o_d[p] = inv_sqrt_df(qh, ql);
                o_I[p] = a.fi ? f2d_nonneg(If[u]) : a.st_I[p + shift];
                o_fo[p] = fs + fo[u];
            }
        }
        for (int f = fams ? f0 : f1; f < f1; f += 32 * kCompactBatch) {
            uint32_t rep[kCompactBatch];
            int mult[kCompactBatch];
#pragma unroll
            for (int u = 0; u < kCompactBatch; u++) {
                const int64_t i = rb + min(f + 32 * u + lane, f1 - 1);
                rep[u] = st_key[i];
                mult[u] = st_mult[i];
            }
#pragma unroll
            for (int u = 0; u < kCompactBatch; u++) {
                const int m = f1 - f - 32 * u;  // families from this 32 on
                if (m <= 0) break;
                if (lane < m) o_mult[fs + f + 32 * u + lane] = mult[u];
                int32_t* __restrict__ out = o_hkl + 3 * (fs + f + 32 * u);
#pragma unroll
                for (int t = 0; t < 3; t++) {
                    const int o = 32 * t + lane, i = o / 3;
                    const uint32_t k = __shfl_sync(0xffffffffu, rep[u], i);
                    if (i < m) out[o] = (int)((k >> (20 - 10 * (o - 3 * i))) & 1023u) - 512;
                }
            }
        }
        P = stop;
    }
}

// Structures of classes c_lo to c_hi, all of at most CAP reflections
template <int CAP, int NT, bool FI>
static void launch_post_class(const PostArgs& a, int c_lo, int c_hi, bool first, bool pdl, cudaStream_t st)
{
    const auto k = k_post<CAP, NT, FI>;
    const size_t smem = post_smem_bytes(CAP);
    static std::atomic<int> per_sm_cache[64] = {};
    int dev = 0;
    cudaGetDevice(&dev);
    int per_sm = (dev >= 0 && dev < 64) ? per_sm_cache[dev].load(std::memory_order_relaxed) : 0;
    if (per_sm < 1) {
        if (smem > 48 * 1024) cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
        // all of the unified L1 / shared storage as shared memory: more structures in flight per SM
        cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared);
        if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k, NT, smem) != cudaSuccess || per_sm < 1) per_sm = 1;
        if (dev >= 0 && dev < 64) per_sm_cache[dev].store(per_sm, std::memory_order_relaxed);
    }
    const int grid = min(a.grid * per_sm, a.n_struct);
    if (pdl) launch_pdl(k, grid, NT, smem, st, a, c_lo, c_hi, first);
    else k<<<grid, NT, smem, st>>>(a, c_lo, c_hi, first);
}

// The size classes in a row on one stream, the largest first, each starting as the CTAs of the one before leave room
// (pdl_chain_enter): the flat passes where a structure can be that large, then the shared-memory classes that a
// structure of the batch can fall into (no structure has more reflections than the batch has room for).
// The classes keep the shared memory of a CTA close to what its structure needs, which matters where structures
// queue for the SMs; a batch that leaves SMs free has nothing to gain from it, and every class costs a launch:
// up to one structure per SM takes one launch for all, up to kPostFewMax structures three. Measured against nine streams
// forked and joined by events, one class each: 24 mixed cells 136 -> 134 us a call, 1024 small cells 247 -> 205 us,
// 256 hexagonal/P1 cells 165 -> 141 us, 20 000 cells at Mo K-alpha 7.38 -> 6.81 ms, rock salt in FP64 155 -> 132 us
// (with the one-launch front, k_front).
constexpr int kPostFewMax = 2048;
template <bool FI>
static void launch_post_fi(const PostArgs& a, int64_t cap_refl, cudaStream_t st, bool pdl)
{
    bool first = true;
    if (cap_refl > kPostCap7) {
        launch_post_flat(a, kPostFlatClass, st);
        first = false;
        pdl = true;
    }
    auto go = [&](auto cap, auto nt, int c_lo, int c_hi, int64_t below) {
        if (c_lo > 0 && cap_refl <= below) return;
        launch_post_class<decltype(cap)::value, decltype(nt)::value, FI>(a, c_lo, c_hi, first, pdl, st);
        first = false;
        pdl = true;
    };
#define XRD_POST(CAP, NT, LO, HI, BELOW) \
    go(std::integral_constant<int, CAP>{}, std::integral_constant<int, NT>{}, LO, HI, BELOW)
    if (a.n_struct <= a.grid && cap_refl > kPostCap3) {
        XRD_POST(kPostCap7, 1024, 0, 7, 0);
    } else if (a.n_struct <= kPostFewMax) {
        XRD_POST(kPostCap7, 1024, 7, 7, kPostCap6);
        XRD_POST(kPostCap6, 512, 4, 6, kPostCap3);
        XRD_POST(kPostCap3, 256, 0, 3, 0);
    } else {
        XRD_POST(kPostCap7, 1024, 7, 7, kPostCap6);
        XRD_POST(kPostCap6, 512, 6, 6, kPostCap5);
        XRD_POST(kPostCap5, 512, 5, 5, kPostCap4);
        XRD_POST(kPostCap4, 256, 4, 4, kPostCap3);
        XRD_POST(kPostCap3, 256, 3, 3, kPostCap2);
        XRD_POST(kPostCap2, 192, 2, 2, kPostCap1);
        XRD_POST(kPostCap1, 128, 1, 1, kPostCap0);
        XRD_POST(kPostCap0, 64, 0, 0, 0);
    }
#undef XRD_POST
}

// With a caller's point group: the family key of every reflection of the batch
// (once per call; the post kernels then compare keys instead of forming orbits).
__global__ void __launch_bounds__(256) k_pg_keys(const PostArgs a, unsigned long long* __restrict__ fkg)
{
    pdl_enter();
    if (*a.abort_flag) return;
    const int64_t total = a.refl_off[a.n_struct];
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < total; r += (int64_t)gridDim.x * blockDim.x)
        fkg[r] = pg_family_key(a.key[r], a.pg, a.npg);
}

void launch_pg_keys(const PostArgs& a, unsigned long long* fkg, cudaStream_t st)
{
    if (a.n_struct > 0 && fkg) launch_pdl(k_pg_keys, a.grid * 8, 256, 0, st, a, fkg);
}

// a.grid = number of SMs
void launch_post(const PostArgs& a, int64_t cap_refl, cudaStream_t st, bool pdl)
{
    if (a.n_struct <= 0) return;
    if (a.If) launch_post_fi<true>(a, cap_refl, st, pdl);
    else launch_post_fi<false>(a, cap_refl, st, pdl);
}

void launch_compact(const CompactArgs& a, cudaStream_t st, bool pdl)
{
    const int nch = (a.n_struct + kOutItems * kOutThreads - 1) / (kOutItems * kOutThreads);
    if (nch <= 2 || !a.parts) {
        if (pdl) launch_pdl(k_scan_out, 1, kOutThreads, 0, st, a);
        else k_scan_out<<<1, kOutThreads, 0, st>>>(a);
    } else {
        k_scan_out_parts<<<nch, kOutThreads, 0, st>>>(a);
        launch_pdl(k_scan_out_final, nch, kOutThreads, 0, st, a);
    }
    if (a.n_struct > 0) launch_pdl(k_compact, a.grid * kCompactCtas, kCompactThreads, 0, st, a);
}

}  // namespace xrd
