// sigma = H x on the CUDA cores in FP64 and FP32, one alpha string (row) per CTA.
//
// With E over unordered orbital pairs s = {p, q} (slots; (pq|rs) is symmetric in
// each pair) the opposite-spin part of the paper's H (Methods) is
//   sum_{s,s'} W[s][s'] E^a_s E^b_s',   W[s][s'] = (pq|rs).
// For one row R (an alpha string), with e over the m(n-m) off-diagonal entries of
// R (target tgt_e, slot s_e, sign g_e) and f over those of a beta string J:
//   D_f(J)    = sum_e g_e W[s_e][s_f] x[tgt_e][J] + vA[s_f][R] x[R][J]
//   y[R][tgt_f(J)] += g_f D_f(J)
// and the beta diagonal entries give y[R][J] += sum_e g_e vB[s_e][J] x[tgt_e][J],
// where v[s][I] = sum_{q in I} W[qq][s] merges a string's m diagonal entries into
// one.  Against one term per ordered table entry (m (n-m+1) squared) that is
// (m (n-m) + 1) squared terms: 1369 instead of 1764 at 12 orbitals.
// x[tgt_e][J] is read along J (coalesced) and W comes from shared memory, so no
// term gathers from global memory.  D goes through shared memory to the thread
// that owns the target: for the k-th entry (t, s) of J', D_f(t) with f the entry of
// t that leads back to J'.  Every sum has a fixed order: the result is the same
// bits on each run, alone or batched.
//
// k_sigma_rows (FP64): thread per (J, group of f); each
// thread computes D only for its string's own entries, so no term is wasted.  At
// FP64 this is what matters: the FP64 pipe takes two FMA per clock and SM (a 64th of the
// FP32 rate), everything else hides behind it.  One column at 12 orbitals: 9.50 ms with a
// thread per determinant (three FP64 operations per pair of table entries), 3.39 ms here
// (1.5 of the two FMA), 2.6 ms at the FP64 rate.
// k_opp_slots / k_same_dense (larger FP32 molecules): see there.  Three columns at 12
// orbitals: 4.33 ms with a thread per determinant (two gathers per FMA), 0.88 ms here.
#include <algorithm>

#include "common.cuh"

namespace kpm {

namespace {

constexpr int ROWS_THREADS = 512;
constexpr size_t SMEM_MAX = 227 * 1024;

__device__ __forceinline__ double flip(double v, uint32_t neg) {
    return __longlong_as_double(__double_as_longlong(v) ^ ((long long)neg << 63));
}
__device__ __forceinline__ float flip(float v, uint32_t neg) {
    return __uint_as_float(__float_as_uint(v) ^ (neg << 31));
}

// ---------------------------------------------------------------- tables

// Off-diagonal entries of each string in table order: target, pair index
// q (q - 1) / 2 + p (p < q) | sign << 15, and the pair index string-fastest.
__global__ void k_off_lists(const int32_t* __restrict__ tgt, const uint16_t* __restrict__ pq,
                            const int8_t* __restrict__ sgn, int64_t ns, int nexc, int noff, int n,
                            int32_t* __restrict__ otgt, uint16_t* __restrict__ oslot,
                            uint16_t* __restrict__ slotT) {
    const int64_t r = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= ns) return;
    int k = 0;
    for (int e = 0; e < nexc; ++e) {
        const int64_t i = r * nexc + e;
        int a = pq[i] / n, b = pq[i] % n;
        if (a == b) continue;
        if (a > b) { const int t = a; a = b; b = t; }
        const int s = b * (b - 1) / 2 + a;
        otgt[r * noff + k] = tgt[i];
        oslot[r * noff + k] = (uint16_t)(s | (sgn[i] < 0 ? 0x8000 : 0));
        slotT[(int64_t)k * ns + r] = (uint16_t)s;
        ++k;
    }
}

// back[r][k]: the entry of string otgt[r][k] that leads back to r (same pair)
__global__ void k_back(const int32_t* __restrict__ otgt, const uint16_t* __restrict__ oslot,
                       int64_t ns, int noff, uint8_t* __restrict__ back) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= ns * noff) return;
    const int64_t t = otgt[i];
    const int s = oslot[i] & 0x7FFF;
    int f = 0;
    while (f < noff && (oslot[t * noff + f] & 0x7FFF) != s) ++f;
    back[i] = (uint8_t)f;
}

// revT[k][r]: r's entries ordered by (back, table order): target | back << 16 |
// sign << 31, string-fastest.
__global__ void k_rev(const int32_t* __restrict__ otgt, const uint16_t* __restrict__ oslot,
                      const uint8_t* __restrict__ back, int64_t ns, int noff,
                      uint32_t* __restrict__ revT) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= ns * noff) return;
    const int64_t r = i / noff;
    const int k = (int)(i - r * noff);
    const int b = back[i];
    int pos = 0;
    for (int j = 0; j < noff; ++j) {
        const int o = back[r * noff + j];
        pos += o < b || (o == b && j < k);
    }
    revT[(int64_t)pos * ns + r] =
        (uint32_t)otgt[i] | ((uint32_t)b << 16) | ((uint32_t)(oslot[i] >> 15) << 31);
}

// stgt[s][r]: target of r under pair s | sign << 15, or ns where there is none
__global__ void k_pair_fill(uint16_t* __restrict__ stgt, int64_t count, int64_t ns) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < count;
         i += (int64_t)gridDim.x * blockDim.x)
        stgt[i] = (uint16_t)ns;
}
__global__ void k_pair_targets(const int32_t* __restrict__ otgt, const uint16_t* __restrict__ oslot,
                               int64_t ns, int noff, uint16_t* __restrict__ stgt) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= ns * noff) return;
    const int64_t r = i / noff;
    const uint16_t w = oslot[i];
    stgt[(int64_t)(w & 0x7FFFu) * ns + r] = (uint16_t)((uint32_t)otgt[i] | (w & 0x8000u));
}

__device__ __forceinline__ void pair_of(int s, int& p, int& q) {
    q = 1;
    while (q * (q + 1) / 2 <= s) ++q;
    p = s - q * (q - 1) / 2;
}

// woo[s][s'] = (pq|rs) over off-diagonal pairs
template <class T>
__global__ void k_woo(const double* __restrict__ eri, int n, int NO, T* __restrict__ woo) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= NO * NO) return;
    int p, q, r, s;
    pair_of(i / NO, p, q);
    pair_of(i % NO, r, s);
    woo[i] = (T)eri[(((int64_t)p * n + q) * n + r) * n + s];
}

// How v is kept: FP64, or float hi + lo (a sum of m integrals rounded once would put
// one systematic error m times as large as an integral's own into H, and the moment
// error grows with the moment index: spectrum error 2e-4 against 4e-5 at 10 orbitals)
__device__ __forceinline__ void store_v(double* v, double s) { *v = s; }
__device__ __forceinline__ void store_v(float2* v, double s) {
    const float h = (float)s;
    *v = make_float2(h, (float)(s - (double)h));
}
__device__ __forceinline__ float v_part(float2 v, int part) { return part ? v.y : v.x; }
// acc + (+-v) a
__device__ __forceinline__ float v_fma(float2 v, uint32_t neg, float a, float acc) {
    return fmaf(flip(v.x, neg), a, fmaf(flip(v.y, neg), a, acc));
}

// v[s][I] = sum_{i in I} (ii|pq) over off-diagonal pairs s = {p, q}
template <class V>
__global__ void k_vdiag(const double* __restrict__ eri, int n, int NO,
                        const uint32_t* __restrict__ masks, int64_t ns, V* __restrict__ v) {
    const int64_t I = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (I >= ns) return;
    int p, q;
    pair_of(blockIdx.y, p, q);
    double s = 0.0;
    for (uint32_t mk = masks[I]; mk; mk &= mk - 1) {
        const int i = __ffs(mk) - 1;
        s += eri[(((int64_t)i * n + i) * n + p) * n + q];
    }
    store_v(v + (int64_t)blockIdx.y * ns + I, s);
}

// c[q][I] = sum_{i in I} (ii|qq)
__global__ void k_cdiag(const double* __restrict__ eri, int n, const uint32_t* __restrict__ masks,
                        int64_t ns, double* __restrict__ c) {
    const int64_t I = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (I >= ns) return;
    const int q = blockIdx.y;
    double s = 0.0;
    for (uint32_t mk = masks[I]; mk; mk &= mk - 1) {
        const int i = __ffs(mk) - 1;
        s += eri[(((int64_t)i * n + i) * n + q) * n + q];
    }
    c[(int64_t)q * ns + I] = s;
}

// Dense off-diagonal string Hamiltonian F [ns][ld], zero where no entry
__global__ void k_dense_f(const int32_t* __restrict__ fcol, const float* __restrict__ fval,
                          int64_t ns, int nnbr, int64_t ld, float* __restrict__ F) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= ns * (nnbr - 1)) return;
    const int64_t t = 1 + i / ns, r = i % ns;
    F[r * ld + fcol[t * ns + r]] = fval[t * ns + r];
}

// ---------------------------------------------------------------- k_sigma_rows

// D of FT entries at a time over the items (group of FT entries, J) of a chunk.
template <int FT>
__device__ __forceinline__ void rows_d_items(const double* x, const double* sB, double* sD,
                                             const uint32_t* rowoff, int K, int kp,
                                             const uint16_t* __restrict__ slotT, int nsb, int f0,
                                             int f1) {
    const int ngrp = (f1 - f0 + FT - 1) / FT;
    for (int w = threadIdx.x; w < nsb * ngrp; w += blockDim.x) {
        const int g = w / nsb, J = w - g * nsb;
        const int fb = f0 + g * FT;
        const double* bp[FT];
        double acc[FT];
#pragma unroll
        for (int i = 0; i < FT; ++i) {
            const int f = min(fb + i, f1 - 1);
            bp[i] = sB + (int)__ldg(slotT + (int64_t)f * nsb + J) * kp;
            acc[i] = 0.0;
        }
        int e = 0;
        for (; e + 4 <= K; e += 4) {
            double a[4];
#pragma unroll
            for (int u = 0; u < 4; ++u) a[u] = x[rowoff[e + u] + J];
#pragma unroll
            for (int u = 0; u < 4; ++u)
#pragma unroll
                for (int i = 0; i < FT; ++i) acc[i] = fma(bp[i][e + u], a[u], acc[i]);
        }
        for (; e < K; ++e) {
            const double a = x[rowoff[e] + J];
#pragma unroll
            for (int i = 0; i < FT; ++i) acc[i] = fma(bp[i][e], a, acc[i]);
        }
#pragma unroll
        for (int i = 0; i < FT; ++i)
            if (fb + i < f1) sD[(fb + i - f0) * nsb + J] = acc[i];
    }
}

// One CTA: alpha string ia, column col.  The opposite-spin sums run over chunks of
// fc entries f (what of D fits in shared memory); the same-spin neighbours and the
// merged beta diagonal are one list of terms per J, in `parts` pieces where a row
// alone would leave threads idle.
__device__ __forceinline__ void sigma_rows_cta(const BatchMol& m, int64_t ia, int64_t col) {
    extern __shared__ __align__(16) unsigned char smem[];
    grid_let_next();
    const int nsb = (int)m.nsb, nsa = (int)m.nsa;
    const int noA = m.noffA, noB = m.noffB, NO = m.NO, K = m.K, kp = m.K | 1;
    const int nfa = m.nnbrA - 1, nfb = m.nnbrB - 1;
    const int64_t dim = m.nsa * m.nsb;
    // (ordinary loads of x: its writer may still run when this CTA starts)
    const double* x = static_cast<const double*>(m.x) + col * dim;
    double* y = static_cast<double*>(m.y) + col * dim;
    // [NO][kp] signed W of this row, read for D only, which strings without an off-diagonal
    // entry do not have
    double* sB = reinterpret_cast<double*>(smem);
    double* sD = sB + (noB > 0 ? (size_t)NO * kp : 0);       // [fc][nsb]
    double* sP = sD + (size_t)m.fc * nsb;                    // [parts][nsb] if parts > 1
    double* sX = sP + (m.parts > 1 ? (size_t)m.parts * nsb : 0);   // [nsb] row of x if staged
    double* sFv = sX + (m.stage_x ? nsb : 0);                // [nfa]
    uint32_t* sFo = reinterpret_cast<uint32_t*>(sFv + nfa);   // [nfa] row offsets
    uint32_t* rowoff = sFo + nfa;                       // [K] offsets of x[tgt_e]
    uint16_t* sS = reinterpret_cast<uint16_t*>(rowoff + K);   // [K] pair | sign << 15
    uint8_t* ptr = reinterpret_cast<uint8_t*>(sS + K);  // [nsb] next entry of the gather
    const double* __restrict__ woo = static_cast<const double*>(m.woo);
    const double* __restrict__ vB = static_cast<const double*>(m.vB);
    const double* __restrict__ fvA = static_cast<const double*>(m.fvalA);
    const double* __restrict__ fvB = static_cast<const double*>(m.fvalB);
    const uint32_t myrow = (uint32_t)ia * (uint32_t)nsb;

    for (int e = threadIdx.x; e < K; e += blockDim.x) {
        // the merged diagonal entry comes last
        rowoff[e] = e < noA ? (uint32_t)m.otgtA[ia * noA + e] * (uint32_t)nsb : myrow;
        sS[e] = e < noA ? m.oslotA[ia * noA + e] : (uint16_t)0;
    }
    for (int t = threadIdx.x; t < nfa; t += blockDim.x) {
        sFv[t] = fvA[(int64_t)(t + 1) * nsa + ia];
        sFo[t] = (uint32_t)m.fcolA[(int64_t)(t + 1) * nsa + ia] * (uint32_t)nsb;
    }
    for (int j = threadIdx.x; j < nsb; j += blockDim.x) ptr[j] = 0;
    __syncthreads();
    for (int i = noB > 0 ? threadIdx.x : NO * K; i < NO * K; i += blockDim.x) {
        const int s = i / K, e = i - s * K;
        sB[s * kp + e] = e < noA ? flip(woo[s * NO + (sS[e] & 0x7FFF)], sS[e] >> 15)
                                 : static_cast<const double*>(m.vA)[(int64_t)s * nsa + ia];
    }
    // x is the previous kernel's output and y may still be its input; all above is tables
    grid_wait();
    if (m.stage_x) {
        for (int j = threadIdx.x; j < nsb; j += blockDim.x) sX[j] = x[myrow + j];
        __syncthreads();
    }

    // terms of J: same-spin beta, same-spin alpha, alpha off-diagonal x beta diagonal
    const int nt = nfb + nfa + noA;
    const double* xr = m.stage_x ? sX : x + myrow;
    for (int w = threadIdx.x; w < nsb * m.parts; w += blockDim.x) {
        const int part = w / nsb, J = w - part * nsb;
        const int t0 = (int)((int64_t)nt * part / m.parts);
        const int t1 = (int)((int64_t)nt * (part + 1) / m.parts);
        double a0 = 0.0, a1 = 0.0;
        int t = t0;
        {
            const int end = min(t1, nfb);
            const double* fv = fvB + nsb + J;
            const int32_t* fc = m.fcolB + nsb + J;
            for (; t + 4 <= end; t += 4) {
                double v[4], xv[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    v[u] = __ldg(fv + (int64_t)(t + u) * nsb);
                    xv[u] = xr[__ldg(fc + (int64_t)(t + u) * nsb)];
                }
                a0 = fma(v[0], xv[0], a0);
                a1 = fma(v[1], xv[1], a1);
                a0 = fma(v[2], xv[2], a0);
                a1 = fma(v[3], xv[3], a1);
            }
            for (; t < end; ++t)
                a0 = fma(__ldg(fv + (int64_t)t * nsb), xr[__ldg(fc + (int64_t)t * nsb)], a0);
        }
        {
            const int end = min(t1, nfb + nfa) - nfb;
            int u = t - nfb;
            for (; u + 4 <= end; u += 4) {
                double xv[4];
#pragma unroll
                for (int i = 0; i < 4; ++i) xv[i] = x[sFo[u + i] + J];
                a0 = fma(sFv[u], xv[0], a0);
                a1 = fma(sFv[u + 1], xv[1], a1);
                a0 = fma(sFv[u + 2], xv[2], a0);
                a1 = fma(sFv[u + 3], xv[3], a1);
            }
            for (; u < end; ++u) a0 = fma(sFv[u], x[sFo[u] + J], a0);
            t = max(t, min(t1, nfb + nfa));
        }
        {
            const int end = t1 - nfb - nfa;
            for (int e = t - nfb - nfa; e < end; ++e) {
                const double v = __ldg(vB + (int64_t)(sS[e] & 0x7FFF) * nsb + J);
                a1 = fma(flip(v, sS[e] >> 15), x[rowoff[e] + J], a1);
            }
        }
        if (m.parts > 1) sP[part * nsb + J] = a0 + a1;
        else y[myrow + J] = a0 + a1;      // read back below by this same thread
    }
    __syncthreads();

    const int nchunk = noB > 0 && K > 0 ? (noB + m.fc - 1) / m.fc : 0;
    for (int c = 0; c < max(nchunk, 1); ++c) {
        const int f0 = c * m.fc, f1 = min(noB, f0 + m.fc);
        if (nchunk) {
            if (m.ft == 6) rows_d_items<6>(x, sB, sD, rowoff, K, kp, m.slotTB, nsb, f0, f1);
            else if (m.ft == 5) rows_d_items<5>(x, sB, sD, rowoff, K, kp, m.slotTB, nsb, f0, f1);
            else rows_d_items<4>(x, sB, sD, rowoff, K, kp, m.slotTB, nsb, f0, f1);
            __syncthreads();
        }
        for (int J = threadIdx.x; J < nsb; J += blockDim.x) {
            double acc;
            if (c == 0) {
                if (m.parts > 1) {
                    acc = sP[J];
                    for (int p = 1; p < m.parts; ++p) acc += sP[p * nsb + J];
                } else {
                    acc = y[myrow + J];
                }
            } else {
                acc = y[myrow + J];
            }
            if (nchunk) {
                int p = nchunk > 1 ? ptr[J] : 0;
                bool more = true;
                while (more && p < noB) {
                    uint32_t wd[8];
#pragma unroll
                    for (int u = 0; u < 8; ++u)
                        wd[u] = __ldg(m.revTB + (int64_t)min(p + u, noB - 1) * nsb + J);
#pragma unroll
                    for (int u = 0; u < 8; ++u) {
                        const int f = (int)((wd[u] >> 16) & 0x7FFFu);
                        more = more && p < noB && f < f1;
                        if (more) {
                            acc += flip(sD[(f - f0) * nsb + (int)(wd[u] & 0xFFFFu)], wd[u] >> 31);
                            ++p;
                        }
                    }
                }
                if (nchunk > 1) ptr[J] = (uint8_t)p;
            }
            if (c + 1 >= nchunk) {
                // the diagonal last: it is the largest term, and every addition after it
                // would round at its size; hi in one rounding with the sum
                {
                    double d = fvA[ia] + fvB[J];
                    for (uint32_t mk = m.maskA[ia]; mk; mk &= mk - 1)
                        d += m.cB[(int64_t)(__ffs(mk) - 1) * nsb + J];
                    acc = fma(d, xr[J], acc);
                }
            }
            y[myrow + J] = acc;
        }
        if (c + 1 < nchunk) __syncthreads();
    }
}

__global__ void __launch_bounds__(ROWS_THREADS, 2)
k_sigma_rows(const __grid_constant__ BatchMol m) {
    sigma_rows_cta(m, blockIdx.x, blockIdx.y);
}

// Batched: the flattened grid covers every molecule's (row, column) CTAs; a CTA
// finds its molecule by binary search over the molecules' first blocks.
__global__ void __launch_bounds__(ROWS_THREADS, 2)
k_sigma_rows_batch(const BatchMol* __restrict__ mols, int nmol) {
    const int64_t blk = blockIdx.x;
    int lo = 0, hi = nmol - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (mols[mid].sblk0 <= blk) lo = mid; else hi = mid - 1;
    }
    const BatchMol& m = mols[lo];
    const int64_t local = blk - m.sblk0;
    sigma_rows_cta(m, local % m.nsa, local / m.nsa);
}

// ---------------------------------------------------------------- k_opp_slots (FP32)

__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
    uint64_t r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void unpack2(uint64_t v, float& lo, float& hi) {
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ void fma2(uint64_t& acc, uint64_t a, uint64_t b) {
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc) : "l"(a), "l"(b));
}

// One determinant in the order of the gather kernel, which touches its neighbours alone.
// The tiled products also multiply by the zeros of the dense F and of padded tables, and an
// infinity or NaN times zero would spread along whole rows and columns: k_opp_slots takes
// every element that came out not finite from here.
__device__ __noinline__ float gather_one(const BatchMol& m, const float* x, int64_t ia,
                                         int64_t ib) {
    const int64_t nsa = m.nsa, nsb = m.nsb;
    const float* fvA = static_cast<const float*>(m.fvalA);
    const float* fvB = static_cast<const float*>(m.fvalB);
    const float* V = static_cast<const float*>(m.V);
    const int n = m.n, n2 = n * n;
    float acc = 0.f;
    for (int t = 1; t < m.nnbrB; ++t)
        acc += fvB[(int64_t)t * nsb + ib] * x[ia * nsb + m.fcolB[(int64_t)t * nsb + ib]];
    for (int t = 1; t < m.nnbrA; ++t)
        acc += fvA[(int64_t)t * nsa + ia] * x[(int64_t)m.fcolA[(int64_t)t * nsa + ia] * nsb + ib];
    for (int f = 0; f < m.nexcB; ++f) {
        const int64_t jb = m.tgtBT[(int64_t)f * nsb + ib];
        const int pb = m.pqBT[(int64_t)f * nsb + ib];
        float inner = 0.f;
        // off-diagonal alpha entries first; diagonal by diagonal is in the exact diagonal
        for (int pass = 0; pass < (pb % (n + 1) == 0 ? 1 : 2); ++pass)
            for (int e = 0; e < m.nexcA; ++e) {
                const int64_t k = ia * m.nexcA + e;
                const int g = m.pqA[k];
                if ((g % (n + 1) == 0) != (pass == 1)) continue;
                inner += float(m.sgnA[k]) * V[(int64_t)g * n2 + pb] *
                         x[(int64_t)m.tgtA[k] * nsb + jb];
            }
        acc += float(m.sgnBT[(int64_t)f * nsb + ib]) * inner;
    }
    const float2 d = m.diag[ia * nsb + ib];
    const float xv = x[ia * nsb + ib];
    return acc + fmaf(d.x, xv, d.y * xv);
}

// Opposite-spin part and diagonal of one row, FP32, added into y.  At FP32 rate one
// shared-memory load per FMA (k_sigma_rows) would bound the row at a quarter of the
// FMA rate or less, so here D is a register-tiled product over all pairs s, whether
// or not a string has them (about half do): TS pairs x TJ columns per thread, W
// rows read as broadcast 16-byte words, x along J one group of four entries ahead,
// two pairs per fma.rn.f32x2.  Passes of TS pairs go through shared memory
// ([TS][nsb + 1], the last cell zero for absent targets) to the thread that owns the
// target.
template <int TS, int TJ, int THREADS>
__global__ void __launch_bounds__(THREADS, 512 / THREADS)
k_opp_slots(const __grid_constant__ BatchMol m) {
    constexpr int TSP = (TS + 3) / 4 * 4, W = 32 * TJ;
    extern __shared__ __align__(16) unsigned char smem[];
    const int nsb = (int)m.nsb, noA = m.noffA, NO = m.NO, K = m.K, ld = nsb + 1;
    const int K4 = (K + 3) / 4 * 4;      // padded with zero rows of W on the own row of x
    const int64_t ia = blockIdx.x, dim = m.nsa * m.nsb;
    const float* __restrict__ x = static_cast<const float*>(m.x) + blockIdx.y * dim;
    float* __restrict__ y = static_cast<float*>(m.y) + blockIdx.y * dim;
    float* sW = reinterpret_cast<float*>(smem);          // [K4][TSP]
    uint32_t* rowoff = reinterpret_cast<uint32_t*>(sW + (size_t)K4 * TSP);  // [K4]
    float* sD = reinterpret_cast<float*>(rowoff + K4);                      // [TS][ld]
    uint16_t* sS = reinterpret_cast<uint16_t*>(sD + (size_t)TS * ld);       // [K4]
    const float* __restrict__ woo = static_cast<const float*>(m.woo);
    const float2* __restrict__ vB = static_cast<const float2*>(m.vB);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const uint32_t myrow = (uint32_t)ia * (uint32_t)nsb;

    for (int e = threadIdx.x; e < K4; e += THREADS) {
        rowoff[e] = e < noA ? (uint32_t)m.otgtA[ia * noA + e] * (uint32_t)nsb : myrow;
        sS[e] = e < noA ? m.oslotA[ia * noA + e] : (uint16_t)0;
    }
    for (int s = threadIdx.x; s < TS; s += THREADS) sD[s * ld + nsb] = 0.f;
    __syncthreads();
    for (int s0 = 0; s0 < NO; s0 += TS) {
        for (int i = threadIdx.x; i < K4 * TSP; i += THREADS) {
            const int e = i / TSP, s = i - e * TSP;
            float w = 0.f;
            if (s < TS && s0 + s < NO && e < K)
                w = e < noA ? flip(woo[(sS[e] & 0x7FFF) * NO + s0 + s], sS[e] >> 15)
                            : v_part(static_cast<const float2*>(m.vA)[(int64_t)(s0 + s) * m.nsa + ia], e - noA);
            sW[i] = w;
        }
        __syncthreads();
        // tiles of W columns; the last one is shifted to end at the row's end (columns
        // it shares with its neighbour come out the same in both)
        for (int t0 = warp * W; t0 < nsb; t0 += THREADS * TJ) {
            const int j0 = min(t0, nsb - W) + lane;
            const float* xj = x + j0;
            uint64_t acc[TJ][TS / 2];
            float ad[TJ];
#pragma unroll
            for (int i = 0; i < TJ; ++i) {
                ad[i] = 0.f;
#pragma unroll
                for (int u = 0; u < TS / 2; ++u) acc[i][u] = 0;
            }
            float a[4][TJ];
            auto fetch = [&](int e) {
                const uint4 o = *reinterpret_cast<const uint4*>(rowoff + e);
#pragma unroll
                for (int i = 0; i < TJ; ++i) {
                    a[0][i] = __ldg(xj + o.x + 32 * i);
                    a[1][i] = __ldg(xj + o.y + 32 * i);
                    a[2][i] = __ldg(xj + o.z + 32 * i);
                    a[3][i] = __ldg(xj + o.w + 32 * i);
                }
            };
            auto step = [&](int e, const float (&c)[4][TJ]) {
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const ulonglong2* w2 = reinterpret_cast<const ulonglong2*>(sW + (e + q) * TSP);
#pragma unroll
                    for (int u = 0; u < TSP / 4; ++u) {
                        const ulonglong2 w = w2[u];
#pragma unroll
                        for (int i = 0; i < TJ; ++i) {
                            const uint64_t aa = pack2(c[q][i], c[q][i]);
                            fma2(acc[i][2 * u], aa, w.x);
                            if (2 * u + 1 < TS / 2) fma2(acc[i][2 * u + 1], aa, w.y);
                        }
                    }
                }
            };
            fetch(0);
            for (int e = 0; e < K4; e += 4) {
                float c[4][TJ];
#pragma unroll
                for (int q = 0; q < 4; ++q)
#pragma unroll
                    for (int i = 0; i < TJ; ++i) c[q][i] = a[q][i];
                if (e + 4 < K4) fetch(e + 4);
                if (s0 == 0) {
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                        if (e + q < noA) {
                            const float2* v = vB + (int64_t)(sS[e + q] & 0x7FFF) * nsb + j0;
                            const uint32_t neg = sS[e + q] >> 15;
#pragma unroll
                            for (int i = 0; i < TJ; ++i) ad[i] = v_fma(__ldg(v + 32 * i), neg, c[q][i], ad[i]);
                        }
                }
                step(e, c);
            }
#pragma unroll
            for (int i = 0; i < TJ; ++i) {
                const int j = j0 + 32 * i;
#pragma unroll
                for (int u = 0; u < TS / 2; ++u) {
                    float lo, hi;
                    unpack2(acc[i][u], lo, hi);
                    sD[(2 * u) * ld + j] = lo;
                    sD[(2 * u + 1) * ld + j] = hi;
                }
                if (s0 == 0 && j >= t0) y[myrow + j] += ad[i];
            }
        }
        __syncthreads();
        const int cnt = min(TS, NO - s0);
        for (int j = threadIdx.x; j < nsb; j += THREADS) {
            const uint16_t* tw = m.stgtB + (int64_t)s0 * nsb + j;
            float acc = 0.f;
#pragma unroll
            for (int s = 0; s < TS; ++s) {
                if (s < cnt) {
                    const uint32_t w = __ldg(tw + (int64_t)s * nsb);
                    acc += flip(sD[s * ld + (int)(w & 0x7FFFu)], w >> 15);
                }
            }
            acc += y[myrow + j];
            if (s0 + TS >= NO) {
                // the diagonal last: every addition after it would round at its size;
                // hi in one rounding with the sum
                const float2 d = m.diag[(int64_t)myrow + j];
                const float xv = __ldg(x + myrow + j);
                acc = fmaf(d.x, xv, fmaf(d.y, xv, acc));
                if (!isfinite(acc)) acc = gather_one(m, x, ia, j);
            }
            y[myrow + j] = acc;
        }
        __syncthreads();
    }
}

// ---------------------------------------------------------------- k_same_dense (FP32)

// Same-spin part of both spins, off-diagonal, FP32, y overwritten:
//   y[R][J] = sum_A F_a[R][A] x[A][J] + sum_B x[R][B] F_b[B][J]
// as one product over the concatenated sum (F is symmetric, so both halves read a
// k-contiguous left and an n-contiguous right operand).  F is 28 % dense at 12
// orbitals and 14 % at 14; the sparse form needs one shared-memory word for every FMA
// (at best 32 FMA per clock and SM, and its neighbour lists on top: 400 us per spin at
// 12 orbitals and 3 columns), the register-tiled dense one runs near the FMA rate.
// BM x BN tiles, 8 x 8 per thread as 4 + 4 rows and columns, two columns per
// fma.rn.f32x2, k-blocks of 16 copied three deep by 4-byte cp.async (rows of x start
// at any multiple of 4 bytes).
constexpr int SS_BK = 16, SS_STAGES = 3;

__device__ __forceinline__ void cp4(float* dst, const float* src, bool ok) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;"
                 ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(ok ? 4u : 0u)
                 : "memory");
}

template <int BM, int BN>
constexpr size_t ss_smem() {
    return (size_t)SS_STAGES * SS_BK * (BM + 4 + BN) * 4;
}

__device__ __forceinline__ void cp16(float* dst, const float* src, bool ok) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;"
                 ::"r"((uint32_t)__cvta_generic_to_shared(dst)), "l"(src), "r"(ok ? 16u : 0u)
                 : "memory");
}

// V4: rows of x start at multiples of 16 bytes (nsb a multiple of 4), so the right
// operand is copied 16 bytes at a time; the left one is transposed on the way and
// always goes 4 bytes at a time.
template <int BM, int BN, bool V4>
__global__ void __launch_bounds__(BM * BN / 64)
k_same_dense(const float* __restrict__ x, float* __restrict__ y, const float* __restrict__ FA,
            int64_t ldA, const float* __restrict__ FB, int64_t ldB, int nsa, int nsb) {
    constexpr int THREADS = BM * BN / 64, LA = BM + 4;
    extern __shared__ __align__(16) unsigned char smem[];
    float* sA = reinterpret_cast<float*>(smem);              // [stages][16][LA], k-major
    float* sB = sA + SS_STAGES * SS_BK * LA;                 // [stages][16][128]
    const int64_t dim = (int64_t)nsa * nsb;
    x += blockIdx.z * dim;
    y += blockIdx.z * dim;
    const int n0 = blockIdx.x * BN, m0 = blockIdx.y * BM;
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // warps of 32 x 64: 4 x 8 threads
    constexpr int WM = BM / 32;
    const int tr = (warp % WM) * 16 + (lane >> 3) * 4, tc = (warp / WM) * 32 + (lane & 7) * 4;
    const int nk1 = (nsa + SS_BK - 1) / SS_BK, nk = nk1 + (nsb + SS_BK - 1) / SS_BK;

    // copies of this thread: left operand, column ka of rows ra + i RS; right operand,
    // columns cb.. of rows kb + i KS
    constexpr int RS = THREADS / SS_BK, NA = BM / RS;
    constexpr int PER = V4 ? BN / 4 : BN, KS = THREADS / PER, NB = SS_BK / KS;
    const int ka = tid % SS_BK, ra = tid / SS_BK;
    const int cb = tid % PER * (V4 ? 4 : 1), kb = tid / PER;
    const bool okc = n0 + cb < nsb;
    auto load = [&](int kt, int st) {
        const bool first = kt < nk1;
        const int k0 = (first ? kt : kt - nk1) * SS_BK, kn = first ? nsa : nsb;
        const int64_t ldl = first ? ldA : nsb, ldr = first ? nsb : ldB;
        const float* L = (first ? FA : x) + (int64_t)(m0 + ra) * ldl + k0 + ka;
        const float* R = (first ? x : FB) + (int64_t)(k0 + kb) * ldr + n0 + cb;
        float* a = sA + st * SS_BK * LA + ka * LA + ra;
        float* b = sB + st * SS_BK * BN + kb * BN + cb;
        const bool okk = k0 + ka < kn;
#pragma unroll
        for (int i = 0; i < NA; ++i) {
            const bool ok = okk && m0 + ra + i * RS < nsa;
            cp4(a + i * RS, ok ? L : x, ok);
            L += RS * ldl;
        }
#pragma unroll
        for (int i = 0; i < NB; ++i) {
            const bool ok = okc && k0 + kb + i * KS < kn;
            if constexpr (V4) cp16(b + i * KS * BN, ok ? R : x, ok);
            else cp4(b + i * KS * BN, ok ? R : x, ok);
            R += KS * ldr;
        }
    };

    uint64_t acc[8][4];
#pragma unroll
    for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = 0;
#pragma unroll
    for (int s = 0; s < SS_STAGES - 1; ++s) {
        if (s < nk) load(s, s);
        asm volatile("cp.async.commit_group;" ::: "memory");
    }
    for (int kt = 0; kt < nk; ++kt) {
        asm volatile("cp.async.wait_group %0;" ::"n"(SS_STAGES - 2) : "memory");
        __syncthreads();
        if (kt + SS_STAGES - 1 < nk) load(kt + SS_STAGES - 1, (kt + SS_STAGES - 1) % SS_STAGES);
        asm volatile("cp.async.commit_group;" ::: "memory");
        const float* a = sA + (kt % SS_STAGES) * SS_BK * LA + tr;
        const float* b = sB + (kt % SS_STAGES) * SS_BK * BN + tc;
#pragma unroll
        for (int k = 0; k < SS_BK; ++k) {
            const float4 a0 = *reinterpret_cast<const float4*>(a + k * LA);
            const float4 a1 = *reinterpret_cast<const float4*>(a + k * LA + BM / 2);
            const ulonglong2 b0 = *reinterpret_cast<const ulonglong2*>(b + k * BN);
            const ulonglong2 b1 = *reinterpret_cast<const ulonglong2*>(b + k * BN + BN / 2);
            const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
#pragma unroll
            for (int i = 0; i < 8; ++i) {
                const uint64_t aa = pack2(av[i], av[i]);
                fma2(acc[i][0], aa, b0.x);
                fma2(acc[i][1], aa, b0.y);
                fma2(acc[i][2], aa, b1.x);
                fma2(acc[i][3], aa, b1.y);
            }
        }
    }
#pragma unroll
    for (int i = 0; i < 8; ++i) {
        const int m = m0 + (i >> 2) * (BM / 2) + tr + (i & 3);
        if (m >= nsa) continue;
        float* row = y + (int64_t)m * nsb;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
            const int n = n0 + (j >> 1) * (BN / 2) + tc + (j & 1) * 2;
            float lo, hi;
            unpack2(acc[i][j], lo, hi);
            if (n < nsb) row[n] = lo;
            if (n + 1 < nsb) row[n + 1] = hi;
        }
    }
}

// ---------------------------------------------------------------- geometry

// the pairs per pass of k_opp_slots that are instantiated, and whether 2 or 4
// columns per thread
constexpr int OPP_TS[] = {26, 24, 22, 20, 18, 16, 14, 12, 8, 4, 2};

size_t opp_smem(int TS, int K, int64_t nsb) {
    const size_t k4 = (size_t)(K + 3) / 4 * 4;
    return k4 * ((TS + 3) / 4 * 4) * 4 + k4 * 4 + (size_t)TS * (nsb + 1) * 4 + k4 * 2 + 16;
}

// Fewest padded pairs plus a per-pass cost (x is read again in each pass), among what
// fits in shared memory; one CTA per SM (no other to compute while it exchanges D)
// counts a quarter more
int opp_choose(int NO, int K, int64_t nsb) {
    int best = 0;
    double cost = 0.0;
    for (int ts : OPP_TS) {
        const size_t sm = opp_smem(ts, K, nsb);
        if (sm > SMEM_MAX) continue;
        const int passes = (NO + ts - 1) / ts;
        const double c = passes * (ts + 5.0) * (2 * sm + 2048 <= SMEM_MAX ? 1.0 : 1.25);
        if (!best || c < cost) {
            best = ts;
            cost = c;
        }
    }
    return best;
}

void rows_geometry(BatchMol& m) {
    const size_t nsb = (size_t)m.nsb;
    const size_t nw = m.noffB > 0 ? (size_t)m.NO * (m.K | 1) : 0;     // signed W
    const size_t fixed = sizeof(double) * (nw + (m.nnbrA - 1)) +
                         4 * (size_t)(m.nnbrA - 1) + 6 * (size_t)m.K + nsb + 32;
    const int noB = m.noffB > 0 ? m.noffB : 1;
    // pieces of the term list: short rows would otherwise leave most threads idle
    m.parts = nsb <= 32 ? 8 : nsb <= 64 ? 6 : nsb <= 128 ? 4 : nsb <= 256 ? 2 : 1;
    m.stage_x = 1;
    auto size = [&](int fc) {
        return fixed + sizeof(double) * nsb * ((size_t)fc + (m.parts > 1 ? m.parts : 0) + m.stage_x);
    };
    m.fc = noB;
    // two CTAs per SM where at least 8 entries a chunk fit, else one
    const size_t half = 112 * 1024;
    if (size(noB) > half) {
        int fc = noB;
        while (fc > 8 && size(fc) > half) --fc;
        if (size(fc) > half) {
            fc = noB;
            while (fc > 1 && size(fc) > SMEM_MAX) --fc;
            if (size(fc) > SMEM_MAX) m.stage_x = 0;
        }
        m.fc = fc;
    }
    // even chunks, and the entries per thread that waste the fewest terms on them
    const int chunks = (noB + m.fc - 1) / m.fc;
    m.fc = (noB + chunks - 1) / chunks;
    int waste = 1 << 30;
    for (int ft : {6, 5, 4}) {
        const int w = (m.fc + ft - 1) / ft * ft;
        if (w < waste) {
            waste = w;
            m.ft = ft;
        }
    }
    m.smem = size(m.fc);
    // A thread per item, and for short rows enough to stage W, 32 entries each, as its 100 KB
    // at 18 orbitals leave room for two CTAs an SM: 18 orbitals, 9 + 1 electrons, 45.3 ms with
    // the 64 threads that 54 items take, 18.4 with 416 (18.5 in the gather kernel); 9 + 0, without
    // W, 10.3 ms with its room kept free and 1.8 without (4.5); 16 orbitals, 8 + 1, 2.64 and 1.63
    const int64_t items = std::max<int64_t>(m.nsb * ((m.fc + m.ft - 1) / m.ft), nw / 32);
    m.threads = (int)(items >= ROWS_THREADS ? ROWS_THREADS : (items + 31) / 32 * 32);
    if (m.threads < 64) m.threads = 64;
}

// (always the same limit: another thread may be about to launch with more)
template <class F>
void set_smem(F* fn, size_t bytes) {
    if (bytes > 48 * 1024)
        KPM_CUDA(cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                      (int)SMEM_MAX));
}

template <int BM, int BN, bool V4>
void launch_same_v(const BatchMol& m, cudaStream_t st) {
    const dim3 grid((unsigned)((m.nsb + BN - 1) / BN), (unsigned)((m.nsa + BM - 1) / BM),
                    (unsigned)m.ncol);
    constexpr size_t smem = ss_smem<BM, BN>();
    set_smem(k_same_dense<BM, BN, V4>, smem);
    k_same_dense<BM, BN, V4><<<grid, BM * BN / 64, smem, st>>>(
        (const float*)m.x, (float*)m.y, m.denseA, m.ldA, m.denseB, m.ldB, (int)m.nsa, (int)m.nsb);
    KPM_LAUNCHED();
}
template <int BM, int BN>
void launch_same(const BatchMol& m, cudaStream_t st) {
    if (m.nsb % 4 == 0 && (reinterpret_cast<uintptr_t>(m.x) & 15) == 0)
        launch_same_v<BM, BN, true>(m, st);
    else
        launch_same_v<BM, BN, false>(m, st);
}

// The tile whose last wave over the SMs wastes the least, in 64 x 64 units
void same_spin(const BatchMol& m, cudaStream_t st) {
    auto cost = [&](int bm, int bn) {
        const int64_t t = (m.nsa + bm - 1) / bm * ((m.nsb + bn - 1) / bn) * m.ncol;
        return (t + m.nsm - 1) / m.nsm * (bm / 64) * (bn / 64);
    };
    const int64_t c44 = cost(128, 128), c24 = cost(64, 128), c22 = cost(64, 64);
    if (c44 <= c24 && c44 <= c22) launch_same<128, 128>(m, st);
    else if (c24 <= c22) launch_same<64, 128>(m, st);
    else launch_same<64, 64>(m, st);
}

template <int TS, int TJ, int THREADS>
void launch_opp(const BatchMol& m, cudaStream_t st) {
    const size_t smem = opp_smem(TS, m.K, m.nsb);
    set_smem(k_opp_slots<TS, TJ, THREADS>, smem);
    k_opp_slots<TS, TJ, THREADS>
        <<<dim3((unsigned)m.nsa, (unsigned)m.ncol), THREADS, smem, st>>>(m);
    KPM_LAUNCHED();
}

// 256 threads where two CTAs fit an SM, else 512
void opp_slots(const BatchMol& m, cudaStream_t st) {
    const bool two = 2 * opp_smem(m.ts, m.K, m.nsb) + 2048 <= SMEM_MAX;
#define KPM_OPP(TS, TJ)                                                                          \
    case TS:                                                                                     \
        if (two) launch_opp<TS, TJ, 256>(m, st); else launch_opp<TS, TJ, 512>(m, st);            \
        break;
    switch (m.ts) {
        KPM_OPP(26, 2)
        KPM_OPP(24, 2)
        KPM_OPP(22, 2)
        KPM_OPP(20, 2)
        KPM_OPP(18, 2)
        KPM_OPP(16, 2)
        KPM_OPP(14, 4)
        KPM_OPP(12, 4)
        KPM_OPP(8, 4)
        KPM_OPP(4, 4)
        KPM_OPP(2, 4)
    }
#undef KPM_OPP
}

}  // namespace

// ---------------------------------------------------------------- host interface

SigmaPath sigma_path(const SpinTables& A, const SpinTables& B, bool f64) {
    // 16-bit targets, 32-bit element offsets
    if (A.ns * B.ns >= ((int64_t)1 << 31) || B.ns > 32767 || A.ns > 65535) return SIGMA_GATHER;
    // A CTA per row: few rows of more than two gather tiles each leave most SMs idle, which
    // the gather kernel's CTA per 128 columns fills.  Gather and row kernels, one column: 16
    // rows of 12870 strings FP64 1.72 and 18.9 ms, FP32 0.40 and 1.47; 12 of 924 FP64 0.107
    // and 0.197, FP32 0.064 and 0.083.  The line is a cautious one: from about 55 rows the row
    // kernels are ahead (55 of 462 FP64 0.181 and 0.140, FP32 0.068 and 0.054; 91 of 3432
    // FP64 3.03 and 1.81, FP32 0.52 and 0.39).
    if (A.ns < 100 && B.ns > 256) return SIGMA_GATHER;
    BatchMol m{};
    sigma_shape(m, A, B, f64);
    if (f64) {
        // Few terms a determinant: its thread in the gather kernel is done before a row's
        // tables are staged.  512 moments, gather and row kernel: (2; 1,1) 10 terms 2.69 and
        // 3.21 ms, (4; 2,1) 34 terms 3.47 and 3.74, (5; 1,1) 35 terms 3.74 both (x, y and z
        // 3.82 and 3.50), (4; 2,2) 48 terms 4.00 and 3.47.  Without opposite-spin entries
        // (8; 4,0) 54 terms 3.21 and 3.47, (10; 5,0) 127 terms 4.52 and 4.25.
        const int terms = m.nexcA * m.nexcB + m.nnbrA + m.nnbrB;
        if (terms < (m.noffB > 0 ? 35 : 64)) return SIGMA_GATHER;
        rows_geometry(m);
        // Chunks of a single entry of D (rows of about 7,000 strings and more) leave three of
        // a thread's four empty and read x again for each: 16 orbitals with 3 + 6 electrons,
        // 8008 strings a row, 90.1 ms against 76.9 in the gather kernel; chunks of two
        // (15 orbitals, 2 + 7) 6.8 ms against 7.8, of six (14, 7 + 7) 76.8 against 224.7
        if (m.fc < 2 && m.fc < m.noffB) return SIGMA_GATHER;
        return m.smem <= SMEM_MAX ? SIGMA_ROWS : SIGMA_GATHER;
    }
    // (Cautious too: the tiled kernels need rows of 128 strings for a tile of theirs.  Gather
    // and tiled, one and three columns: 462 strings, 11 orbitals, 0.348 and 0.115, 0.858 and
    // 0.207 ms; 252 strings, 10 orbitals, 0.091 and 0.047, 0.188 and 0.075; 210 strings 0.072
    // and 0.045, 0.153 and 0.070.  The dense F pays at every size measured, though it has up
    // to 28 times the neighbours' terms: 18 orbitals, 9 + 3, 160 and 102 ms; 17 orbitals, 7 + 3,
    // 43.9 and 18.9; 16 orbitals, 6 + 6, 250 and 92.)
    if (B.ns <= 300) return SIGMA_GATHER;
    return m.K > 0 && m.NO > 0 && m.noffB > 0 && opp_choose(m.NO, m.K, m.nsb)
               ? SIGMA_SLOTS
               : SIGMA_GATHER;
}

void sigma_shape(BatchMol& m, const SpinTables& A, const SpinTables& B, bool f64) {
    m.nsa = A.ns;
    m.nsb = B.ns;
    m.nexcA = A.nexc;
    m.nexcB = B.nexc;
    m.nnbrA = A.nnbr;
    m.nnbrB = B.nnbr;
    m.n = A.n;
    m.noffA = A.m * (A.n - A.m);
    m.noffB = B.m * (B.n - B.m);
    m.NO = A.n * (A.n - 1) / 2;
    m.K = A.m > 0 ? m.noffA + (f64 ? 1 : 2) : 0;
}

void PairTables::build_spin(Spin& t, const SpinTables& T, const double* eri, SigmaPath path, bool f64,
                            cudaStream_t st) {
    const int noff = T.m * (T.n - T.m), NO = T.n * (T.n - 1) / 2;
    const int64_t ne = T.ns * noff;
    const unsigned bs = (unsigned)((T.ns + 127) / 128);
    t.otgt.alloc((size_t)ne * 4 + 4);
    t.oslot.alloc((size_t)ne * 2 + 4);
    t.slotT.alloc((size_t)ne * 2 + 4);
    t.v.alloc((size_t)NO * T.ns * 8 + 8);
    if (NO > 0) {
        const dim3 g(bs, (unsigned)NO);
        if (f64) k_vdiag<double><<<g, 128, 0, st>>>(eri, T.n, NO, T.masks.as<uint32_t>(), T.ns, t.v.as<double>());
        else k_vdiag<float2><<<g, 128, 0, st>>>(eri, T.n, NO, T.masks.as<uint32_t>(), T.ns, t.v.as<float2>());
        KPM_LAUNCHED();
    }
    if (ne > 0) {
        k_off_lists<<<bs, 128, 0, st>>>(T.tgt.as<int32_t>(), T.pq.as<uint16_t>(), T.sgn.as<int8_t>(),
                                        T.ns, T.nexc, noff, T.n, t.otgt.as<int32_t>(),
                                        t.oslot.as<uint16_t>(), t.slotT.as<uint16_t>());
        KPM_LAUNCHED();
    }
    const unsigned be = (unsigned)((ne + 127) / 128);
    if (path == SIGMA_ROWS && ne > 0) {
        t.back.alloc((size_t)ne);
        t.revT.alloc((size_t)ne * 4);
        k_back<<<be, 128, 0, st>>>(t.otgt.as<int32_t>(), t.oslot.as<uint16_t>(), T.ns, noff,
                                   t.back.as<uint8_t>());
        KPM_LAUNCHED();
        k_rev<<<be, 128, 0, st>>>(t.otgt.as<int32_t>(), t.oslot.as<uint16_t>(),
                                  t.back.as<uint8_t>(), T.ns, noff, t.revT.as<uint32_t>());
        KPM_LAUNCHED();
    }
    if (path == SIGMA_ROWS && f64) {
        t.c.alloc((size_t)T.n * T.ns * 8);
        k_cdiag<<<dim3(bs, (unsigned)T.n), 128, 0, st>>>(eri, T.n, T.masks.as<uint32_t>(), T.ns,
                                                         t.c.as<double>());
        KPM_LAUNCHED();
    }
    if (path == SIGMA_SLOTS) {
        const int64_t np = (int64_t)NO * T.ns;
        t.stgt.alloc((size_t)np * 2);
        k_pair_fill<<<1024, 256, 0, st>>>(t.stgt.as<uint16_t>(), np, T.ns);
        KPM_LAUNCHED();
        if (ne > 0) {
            k_pair_targets<<<be, 128, 0, st>>>(t.otgt.as<int32_t>(), t.oslot.as<uint16_t>(), T.ns,
                                               noff, t.stgt.as<uint16_t>());
            KPM_LAUNCHED();
        }
        t.ld = (T.ns + 3) / 4 * 4;
        t.dense.alloc((size_t)T.ns * t.ld * 4);
        KPM_CUDA(cudaMemsetAsync(t.dense.p, 0, t.dense.bytes, st));
        const int64_t nf = T.ns * (int64_t)(T.nnbr - 1);
        if (nf > 0) {
            k_dense_f<<<(unsigned)((nf + 255) / 256), 256, 0, st>>>(
                T.fcol.as<int32_t>(), T.fval32.as<float>(), T.ns, T.nnbr, t.ld,
                t.dense.as<float>());
            KPM_LAUNCHED();
        }
    }
}

size_t PairTables::bytes(const SpinTables& A, const SpinTables& B, bool f64, bool dense) {
    const SigmaPath path = sigma_path(A, B, f64);
    if (path == SIGMA_GATHER || (path == SIGMA_SLOTS && !dense)) return 0;
    const size_t NO = A.n * (A.n - 1) / 2;
    // as build_spin allocates
    auto spin = [&](const SpinTables& T) {
        const size_t ns = T.ns, ne = ns * T.m * (T.n - T.m);
        const size_t common = 8 * ne + 8 * NO * ns;
        return path == SIGMA_ROWS ? common + 5 * ne + 8 * T.n * ns
                                  : common + 2 * NO * ns + 4 * ns * ((ns + 3) / 4 * 4);
    };
    return NO * NO * (f64 ? 8 : 4) + spin(A) + (&A != &B ? spin(B) : 0);
}

void PairTables::build(const SpinTables& A, const SpinTables& B, const double* eri, bool f64_,
                       cudaStream_t st) {
    f64 = f64_;
    int dev = 0;
    KPM_CUDA(cudaGetDevice(&dev));
    KPM_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
    path = sigma_path(A, B, f64);
    if (path == SIGMA_GATHER) return;
    try {
        build_tables(A, B, eri, st);
    } catch (const Error& e) {
        // no memory for the row kernels' tables (the dense F of 48620 strings is 9.5 GB, five
        // times everything else that such a context holds): the gather kernel needs none
        if (e.status != KPM_ENOMEM) throw;
        KPM_CUDA(cudaStreamSynchronize(st));
        woo.release();
        a.release();
        b_own.release();
        b = nullptr;
        path = SIGMA_GATHER;
    }
}

void PairTables::build_tables(const SpinTables& A, const SpinTables& B, const double* eri,
                              cudaStream_t st) {
    const int NO = A.n * (A.n - 1) / 2;
    woo.alloc((size_t)NO * NO * (f64 ? 8 : 4) + 8);
    if (NO > 0) {
        const unsigned g = (unsigned)((NO * NO + 127) / 128);
        if (f64) k_woo<double><<<g, 128, 0, st>>>(eri, A.n, NO, woo.as<double>());
        else k_woo<float><<<g, 128, 0, st>>>(eri, A.n, NO, woo.as<float>());
        KPM_LAUNCHED();
    }
    build_spin(a, A, eri, path, f64, st);
    if (&A != &B) build_spin(b_own, B, eri, path, f64, st);
    b = &A != &B ? &b_own : &a;
}

void PairTables::fill(BatchMol& m) const {
    m.path = path;
    if (path == SIGMA_GATHER) return;
    m.otgtA = a.otgt.as<int32_t>();
    m.oslotA = a.oslot.as<uint16_t>();
    m.slotTB = b->slotT.as<uint16_t>();
    m.revTB = b->revT.as<uint32_t>();
    m.stgtB = b->stgt.as<uint16_t>();
    m.woo = woo.p;
    m.vA = a.v.p;
    m.vB = b->v.p;
    m.cB = b->c.as<double>();
    m.denseA = a.dense.as<float>();
    m.denseB = b->dense.as<float>();
    m.ldA = a.ld;
    m.ldB = b->ld;
    m.nsm = nsm;
    if (path == SIGMA_SLOTS) m.ts = opp_choose(m.NO, m.K, m.nsb);
    else rows_geometry(m);
}

void sigma_rows(const BatchMol& m, cudaStream_t st) {
    if (m.ncol <= 0 || m.nsa * m.nsb == 0) return;
    if (m.path == SIGMA_SLOTS) {
        same_spin(m, st);
        opp_slots(m, st);
        return;
    }
    const dim3 grid((unsigned)m.nsa, (unsigned)m.ncol);
    set_smem(k_sigma_rows, m.smem);
    launch_chained(k_sigma_rows, grid, m.threads, m.smem, st, m);
    KPM_LAUNCHED();
}

void sigma_rows_batch(const BatchMol* mols, int nmol, int64_t blocks, size_t smem, int threads,
                      cudaStream_t st) {
    if (nmol <= 0 || blocks <= 0) return;
    if (blocks > 0x7FFFFFFFLL) KPM_THROW(KPM_EINVAL, "batched sigma grid too large");
    set_smem(k_sigma_rows_batch, smem);
    k_sigma_rows_batch<<<(unsigned)blocks, threads, smem, st>>>(mols, nmol);
    KPM_LAUNCHED();
}

}  // namespace kpm
