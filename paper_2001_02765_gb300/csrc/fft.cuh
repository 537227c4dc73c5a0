// Shared-memory Stockham FFT, executed by a whole CTA, for lengths 2^k, 3 2^k and
// 5 2^k.
//
// NB independent sequences of length L lie back to back in shared memory
// (element k of sequence s at logical index s * L + k, see spad below). Each stage of radix R reads the
// R inputs of every butterfly into registers, synchronises, applies the
// twiddles and a radix-R DFT in registers and writes the outputs to their
// auto-sorted positions, then synchronises again; one buffer therefore serves
// every stage. Radix 8 is used while at least 8 points remain per sub-transform,
// then one radix-4 or radix-2 stage; a factor 3 or 5 goes into the second stage,
// alone or with factors of two so that the stages are as few as possible
// (768 = 8 x 12 x 8, 640 = 8 x 10 x 8, 1536 = 8 x 3 x 8 x 8; see stage_radix).
//
// Stage with span NS (product of the radices before it) and radix R, for the
// butterfly j in [0, L/R) of a sequence, k = j mod NS:
//     v_r = x[j + r L/R] * W_{NS R}^{r k},   r = 0..R-1
//     X = DFT_R(v)
//     y[(j / NS) NS R + k + r NS] = X_r
// (the Stockham auto-sort formulation; the output is in natural order).
//
// Twiddles: a compact table per length L holds, for every stage with span
// NS > 1, the NS values W_{NS R}^k = exp(-2 pi i k / (NS R)), k < NS, built in
// FP64 on the device (sincospi) and cast for FP32 plans; the stages' tables lie
// back to back. A butterfly loads W^k once (consecutive k: a coalesced load)
// and forms W^{2k} .. W^{(R-1)k} by complex products of depth at most 3 (4 above
// W^{8k}). The inverse transform uses the conjugates and is not normalised.
//
// Shared-memory layout: element i of the batch is stored at spad(i), which
// inserts one padding element every 16 (8-byte complex) or 8 (16-byte complex)
// elements so that the strided stores of the early stages fall in distinct
// banks (for a warp, about 1.1x the conflict-free wavefront count instead of
// 2x). Every access to an FFT buffer goes through spad; spad_size(n) is the
// number of elements a buffer holding n logical elements needs.
#pragma once

#include "common.cuh"

template <typename C>
__host__ __device__ __forceinline__ constexpr int spad(int i)
{
    return sizeof(C) == 8 ? i + (i >> 4) : i + (i >> 3);
}

// elements per padding group: spad(i + g m) = spad(i) + m spad(g) for whole groups
template <typename C>
__host__ __device__ __forceinline__ constexpr int spad_group()
{
    return sizeof(C) == 8 ? 16 : 8;
}

template <typename C>
__host__ __device__ __forceinline__ constexpr int spad_size(int n)
{
    return spad<C>(n - 1) + 1;
}

template <typename C, bool INV>
__device__ __forceinline__ C twiddle(const C *__restrict__ tw, int idx)
{
    C w = __ldg(&tw[idx]);
    if (INV) w.y = -w.y;
    return w;
}

// Odd factor of a length 2^k, 3 2^k or 5 2^k.
__host__ __device__ constexpr int odd_part(int L)
{
    while (L % 2 == 0) L /= 2;
    return L;
}

// Radix of the stage of span NS of a length-L transform. First 8 (the register
// form needs it); then, for L = 3 2^k or 5 2^k, the odd factor with as many
// factors of two as leave whole radix-8 stages (6, 10, 12; radix 20 is left to a
// last radix-4 stage); then 8s and a last 8, 4 or 2.
__host__ __device__ constexpr int stage_radix(int L, int NS)
{
    const int rem = L / NS, m = odd_part(L);
    if (NS == 8 && m > 1) {
        int e = 0;
        for (int r = rem / m; r > 1; r /= 2) ++e;  // rem = m 2^e
        if (e % 3 == 1) return 2 * m;
        if (e % 3 == 2 && m == 3) return 4 * m;
        return m;
    }
    return rem >= 8 ? 8 : rem;
}

// offset of the table of the stage of span NS in a length-L transform's compact table
__host__ __device__ constexpr int stage_table_offset(int L, int NS)
{
    int off = 0;
    for (int ns = 1; ns < NS; ns *= stage_radix(L, ns))
        if (ns > 1) off += ns;
    return off;
}

// entries of the compact table of a length-L transform
__host__ __device__ constexpr int stage_table_size(int L) { return stage_table_offset(L, L); }

// multiply by -i (forward) or +i (inverse)
template <typename C, bool INV>
__device__ __forceinline__ C rot90(C a)
{
    return INV ? cmake<C>(-a.y, a.x) : cmake<C>(a.y, -a.x);
}

template <typename C, bool INV>
__device__ __forceinline__ void dft2(C &a, C &b)
{
    C t = a;
    a = cadd(t, b);
    b = csub(t, b);
}

template <typename C, bool INV>
__device__ __forceinline__ void dft4(C &v0, C &v1, C &v2, C &v3)
{
    C t0 = cadd(v0, v2), t1 = csub(v0, v2);
    C t2 = cadd(v1, v3), t3 = rot90<C, INV>(csub(v1, v3));
    v0 = cadd(t0, t2);
    v2 = csub(t0, t2);
    v1 = cadd(t1, t3);
    v3 = csub(t1, t3);
}

template <typename C, bool INV>
__device__ __forceinline__ void dft8(C *v)
{
    using T = decltype(C::x);
    const T s = (T)0.70710678118654752440;  // 1/sqrt(2)
    C e0 = v[0], e1 = v[2], e2 = v[4], e3 = v[6];
    C o0 = v[1], o1 = v[3], o2 = v[5], o3 = v[7];
    dft4<C, INV>(e0, e1, e2, e3);
    dft4<C, INV>(o0, o1, o2, o3);
    // o_k *= W8^k, W8 = exp(-+ 2 pi i / 8)
    C w1 = INV ? cmake<C>(s * (o1.x - o1.y), s * (o1.x + o1.y)) : cmake<C>(s * (o1.x + o1.y), s * (o1.y - o1.x));
    C w2 = rot90<C, INV>(o2);
    C w3 = INV ? cmake<C>(-s * (o3.x + o3.y), s * (o3.x - o3.y)) : cmake<C>(s * (o3.y - o3.x), -s * (o3.x + o3.y));
    v[0] = cadd(e0, o0);
    v[4] = csub(e0, o0);
    v[1] = cadd(e1, w1);
    v[5] = csub(e1, w1);
    v[2] = cadd(e2, w2);
    v[6] = csub(e2, w2);
    v[3] = cadd(e3, w3);
    v[7] = csub(e3, w3);
}

template <typename C, bool INV>
__device__ __forceinline__ void dft3(C &v0, C &v1, C &v2)
{
    using T = decltype(C::x);
    const T h = (T)0.86602540378443864676;  // sin(2 pi / 3)
    const C t = cadd(v1, v2);
    const C d = rot90<C, INV>(csub(v1, v2));
    const C u = cmake<C>(fma((T)-0.5, t.x, v0.x), fma((T)-0.5, t.y, v0.y));
    v0 = cadd(v0, t);
    v1 = cmake<C>(fma(h, d.x, u.x), fma(h, d.y, u.y));
    v2 = cmake<C>(fma(-h, d.x, u.x), fma(-h, d.y, u.y));
}

template <typename C, bool INV>
__device__ __forceinline__ void dft5(C &v0, C &v1, C &v2, C &v3, C &v4)
{
    using T = decltype(C::x);
    const T c1 = (T)0.30901699437494742410, c2 = (T)-0.80901699437494742410;  // cos(2 pi / 5), cos(4 pi / 5)
    const T s1 = (T)0.95105651629515357212, s2 = (T)0.58778525229247312917;   // sin(2 pi / 5), sin(4 pi / 5)
    const C a = cadd(v1, v4), b = cadd(v2, v3);
    const C d = rot90<C, INV>(csub(v1, v4)), e = rot90<C, INV>(csub(v2, v3));
    const C p = cmake<C>(fma(c1, a.x, fma(c2, b.x, v0.x)), fma(c1, a.y, fma(c2, b.y, v0.y)));
    const C q = cmake<C>(fma(c2, a.x, fma(c1, b.x, v0.x)), fma(c2, a.y, fma(c1, b.y, v0.y)));
    const C r = cmake<C>(fma(s1, d.x, s2 * e.x), fma(s1, d.y, s2 * e.y));
    const C w = cmake<C>(fma(s2, d.x, -s1 * e.x), fma(s2, d.y, -s1 * e.y));
    v0 = cadd(v0, cadd(a, b));
    v1 = cadd(p, r);
    v4 = csub(p, r);
    v2 = cadd(q, w);
    v3 = csub(q, w);
}

// DFT of R points. 6 = 2 x 3, 10 = 2 x 5 and 12 = 4 x 3 by the prime-factor
// mapping (input N2 n1 + N1 n2, output by the remainders: no inner twiddles).
template <typename C, int R, bool INV>
__device__ __forceinline__ void dft(C *v)
{
    if constexpr (R == 8) dft8<C, INV>(v);
    else if constexpr (R == 4) dft4<C, INV>(v[0], v[1], v[2], v[3]);
    else if constexpr (R == 2) dft2<C, INV>(v[0], v[1]);
    else if constexpr (R == 3) dft3<C, INV>(v[0], v[1], v[2]);
    else if constexpr (R == 5) dft5<C, INV>(v[0], v[1], v[2], v[3], v[4]);
    else {
        static_assert(R == 6 || R == 10 || R == 12, "radix");
        constexpr int N1 = R == 12 ? 4 : 2, N2 = R / N1;
        constexpr int e1 = R == 12 ? 9 : N2;          // 1 mod N1, 0 mod N2
        constexpr int e2 = R == 6 ? 4 : (R == 10 ? 6 : 4);  // 0 mod N1, 1 mod N2
        C t[N1][N2];
#pragma unroll
        for (int i = 0; i < N1; ++i)
#pragma unroll
            for (int j = 0; j < N2; ++j) t[i][j] = v[(N2 * i + N1 * j) % R];
#pragma unroll
        for (int i = 0; i < N1; ++i) {
            if constexpr (N2 == 3) dft3<C, INV>(t[i][0], t[i][1], t[i][2]);
            else dft5<C, INV>(t[i][0], t[i][1], t[i][2], t[i][3], t[i][4]);
        }
#pragma unroll
        for (int j = 0; j < N2; ++j) {
            if constexpr (N1 == 2) dft2<C, INV>(t[0][j], t[1][j]);
            else dft4<C, INV>(t[0][j], t[1][j], t[2][j], t[3][j]);
        }
#pragma unroll
        for (int i = 0; i < N1; ++i)
#pragma unroll
            for (int j = 0; j < N2; ++j) v[(e1 * i + e2 * j) % R] = t[i][j];
    }
}

// v[r] *= w1^r, the powers formed by products
template <typename C, int R>
__device__ __forceinline__ void twiddle_powers(C *v, C w1)
{
    v[1] = cmul(v[1], w1);
    if constexpr (R >= 3) {
        const C w2 = cmul(w1, w1);
        v[2] = cmul(v[2], w2);
        if constexpr (R >= 4) {
            const C w3 = cmul(w2, w1);
            v[3] = cmul(v[3], w3);
            if constexpr (R >= 5) {
                const C w4 = cmul(w2, w2);
                v[4] = cmul(v[4], w4);
                if constexpr (R >= 6) {
                    const C w5 = cmul(w4, w1);
                    v[5] = cmul(v[5], w5);
                    if constexpr (R >= 8) {
                        v[6] = cmul(v[6], cmul(w3, w3));
                        v[7] = cmul(v[7], cmul(w4, w3));
                        if constexpr (R >= 10) {
                            v[8] = cmul(v[8], cmul(w4, w4));
                            v[9] = cmul(v[9], cmul(w5, w4));
                            if constexpr (R >= 12) {
                                v[10] = cmul(v[10], cmul(w5, w5));
                                v[11] = cmul(v[11], cmul(cmul(w3, w3), w5));
                            }
                        }
                    }
                }
            }
        }
    }
}

// IN_HALF: the first stage takes the inputs at logical positions >= L/2 as
// zero without reading them (zero padding to at least twice the data length).
// OUT_HALF: the last stage writes only the outputs at positions < L/2.
template <typename C, int L, int NB, int THREADS, int NS, int R, bool INV, bool IN_HALF, bool OUT_HALF, int SEQ>
__device__ __forceinline__ void fft_stage(C *buf, const C *__restrict__ tw)
{
    constexpr int NBF = NB * (L / R);            // butterflies in the stage
    constexpr int PER = (NBF + THREADS - 1) / THREADS;
    C v[PER][R];
    // the R inputs of a butterfly lie L/R apart; when L/R is a whole number of
    // padding groups their padded positions lie a constant distance apart too
    constexpr int S = L / R;
    constexpr bool SPAN_IN = S % spad_group<C>() == 0;
#pragma unroll
    for (int p = 0; p < PER; ++p) {
        const int b = threadIdx.x + p * THREADS;
        if (NBF % THREADS == 0 || b < NBF) {
            const int seq = b / S, j = b % S;
            const C *src = buf + seq * SEQ;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (IN_HALF && NS == 1 && r >= R / 2) v[p][r] = cmake<C>(0, 0);
                else if constexpr (SPAN_IN) v[p][r] = src[spad<C>(j) + r * spad<C>(S)];
                else v[p][r] = src[spad<C>(j + r * S)];
            }
        }
    }
    __syncthreads();
#pragma unroll
    for (int p = 0; p < PER; ++p) {
        const int b = threadIdx.x + p * THREADS;
        if (NBF % THREADS == 0 || b < NBF) {
            const int seq = b / (L / R), j = b % (L / R);
            const int k = j % NS;
            if constexpr (NS > 1) twiddle_powers<C, R>(v[p], twiddle<C, INV>(tw, stage_table_offset(L, NS) + k));
            dft<C, R, INV>(v[p]);
            const int base = (j / NS) * NS * R + k;
            constexpr bool SPAN_OUT = NS % spad_group<C>() == 0;
            C *dst = buf + seq * SEQ;
#pragma unroll
            for (int r = 0; r < R; ++r) {
                if (OUT_HALF && NS * R == L && r >= R / 2) continue;  // position k + r NS >= L/2
                if constexpr (SPAN_OUT) dst[spad<C>(base) + r * spad<C>(NS)] = v[p][r];
                else dst[spad<C>(base + r * NS)] = v[p][r];
            }
        }
    }
    __syncthreads();
}

template <typename C, int L, int NB, int THREADS, int NS, bool INV, bool IN_HALF, bool OUT_HALF, int SEQ>
__device__ __forceinline__ void fft_stages(C *buf, const C *__restrict__ tw)
{
    if constexpr (NS < L) {
        constexpr int R = stage_radix(L, NS);
        fft_stage<C, L, NB, THREADS, NS, R, INV, IN_HALF, OUT_HALF, SEQ>(buf, tw);
        fft_stages<C, L, NB, THREADS, NS * R, INV, IN_HALF, OUT_HALF, SEQ>(buf, tw);
    }
}

// FFT of NB sequences of length L in shared memory by THREADS threads.
// Must be called by every thread of the CTA (it synchronises). The caller
// synchronises before the call so that the inputs are visible. With IN_HALF
// the inputs at positions >= L/2 are taken as zero (and need not be written);
// with OUT_HALF only the outputs at positions < L/2 are produced. SEQ: elements
// from one sequence to the next (default: back to back, spad(s L + k) = s spad(L) + spad(k)).
template <typename C, int L, int NB, int THREADS, bool INV, bool IN_HALF = false, bool OUT_HALF = false,
          int SEQ = spad<C>(L)>
__device__ __forceinline__ void fft_batch(C *buf, const C *__restrict__ tw)
{
    fft_stages<C, L, NB, THREADS, 1, INV, IN_HALF, OUT_HALF, SEQ>(buf, tw);
}

// ------------------------------------------------- register-resident form --
//
// The same stages with the data kept in registers between them, for CTAs of
// NSEQ * L / 8 threads (eight elements per thread). Thread t works on sequence
// seq = t / (L/8) and holds, at the start and at the end of a transform, the
// elements of the "pattern P0": v[m] = element jt + m L/8 of its sequence,
// jt = t mod (L/8), m = 0..7. That is the input pattern of a radix-8 first
// stage (butterfly j = jt reads j + r L/8) and the output pattern of the last
// stage (butterfly j writes j + r NS with NS = L/R; a last stage of radix R < 8
// gives thread t the butterflies jt + p L/8, p < 8/R, so that its outputs are
// again P0). Consequences: a transform needs no shared memory before its first
// stage or after its last (loads and stores to global memory go straight to
// and from registers), a forward transform's outputs are the inputs of an
// inverse transform of the same thread with no exchange in between, and
// between two stages one exchange through shared memory (outputs written to
// their auto-sorted positions, a barrier, next inputs read). With NBUF = 2 the
// exchanges alternate between two buffers (one barrier each; `par` carries the
// buffer parity from one transform to the next); with NBUF = 1 a second
// barrier separates each exchange's reads from the next one's writes. Every
// butterfly does the arithmetic of fft_stage (same twiddles, same radix-R
// DFT), so the results are those of fft_batch.
//
// A middle stage of radix 3, 5, 6, 10 or 12 has L/R butterflies for the L/8
// threads of a sequence: its inputs and outputs go through the exchanges anyway,
// so a thread takes butterflies jt, jt + L/8, ... below L/R. Threads beyond
// NSEQ L / 8 only join the barriers.
template <typename C, int L, int NSEQ, int THREADS, int NS, int NBUF, bool INV, int SEQ>
__device__ __forceinline__ void rfft_stages(C (&v)[8], C *bufs, int &par, const C *__restrict__ tw)
{
    static_assert(THREADS >= NSEQ * L / 8, "eight elements per thread");
    if constexpr (NS < L) {
        constexpr int R = stage_radix(L, NS);
        constexpr bool EVEN = 8 % R == 0;    // whole butterflies of the thread's eight elements
        constexpr int PER = (8 + R - 1) / R;
        constexpr int S = L / R;
        constexpr int BUF = SEQ == spad<C>(L) ? spad_size<C>(NSEQ * L) : NSEQ * SEQ;
        constexpr bool ALL = THREADS == NSEQ * L / 8;
        const int seq = threadIdx.x / (L / 8), jt = threadIdx.x % (L / 8);
        const bool live = ALL || seq < NSEQ;
        if constexpr (!EVEN && NBUF == 2) {
            // from one buffer to the other, a butterfly at a time (fewer registers)
            const C *in = bufs + (par ^ 1) * BUF;
            C *out = bufs + par * BUF;
#pragma unroll
            for (int p = 0; p < PER; ++p) {
                const int j = jt + p * (L / 8);
                if (!(live && j < S)) continue;
                C u[R];
#pragma unroll
                for (int r = 0; r < R; ++r) u[r] = in[seq * SEQ + spad<C>(j + r * S)];
                twiddle_powers<C, R>(u, twiddle<C, INV>(tw, stage_table_offset(L, NS) + j % NS));
                dft<C, R, INV>(u);
                const int base = (j / NS) * NS * R + j % NS;
#pragma unroll
                for (int r = 0; r < R; ++r) out[seq * SEQ + spad<C>(base + r * NS)] = u[r];
            }
            __syncthreads();
            par ^= 1;
            rfft_stages<C, L, NSEQ, THREADS, NS * R, NBUF, INV, SEQ>(v, bufs, par, tw);
            return;
        }
        C u[PER * R];
        if constexpr (NS == 1) {
            static_assert(NS > 1 || R == 8, "first stage");
#pragma unroll
            for (int m = 0; m < 8; ++m) u[m] = v[m];
        } else {
            // gather this stage's inputs from the previous stage's outputs
            const C *in = bufs + (NBUF == 2 ? (par ^ 1) * BUF : 0);
#pragma unroll
            for (int p = 0; p < PER; ++p) {
                const int j = jt + p * (L / 8);
                if (!(live && (EVEN || j < S))) continue;
#pragma unroll
                for (int r = 0; r < R; ++r) u[p * R + r] = in[seq * SEQ + spad<C>(j + r * S)];
            }
            if constexpr (NBUF == 1) __syncthreads();
        }
#pragma unroll
        for (int p = 0; p < PER; ++p) {
            const int j = jt + p * (L / 8);
            if (!(live && (EVEN || j < S))) continue;
            if constexpr (NS > 1)
                twiddle_powers<C, R>(u + p * R, twiddle<C, INV>(tw, stage_table_offset(L, NS) + j % NS));
            dft<C, R, INV>(u + p * R);
        }
        if constexpr (NS * R == L) {
            // last stage: butterfly jt + p L/8, output r at jt + (p + r PER) L/8
            static_assert(EVEN, "last stage");
#pragma unroll
            for (int p = 0; p < PER; ++p)
#pragma unroll
                for (int r = 0; r < R; ++r) v[p + r * PER] = u[p * R + r];
        } else {
            C *out = bufs + (NBUF == 2 ? par * BUF : 0);
#pragma unroll
            for (int p = 0; p < PER; ++p) {
                const int j = jt + p * (L / 8);
                if (!(live && (EVEN || j < S))) continue;
                const int base = (j / NS) * NS * R + j % NS;
#pragma unroll
                for (int r = 0; r < R; ++r) out[seq * SEQ + spad<C>(base + r * NS)] = u[p * R + r];
            }
            __syncthreads();
            if constexpr (NBUF == 2) par ^= 1;
            rfft_stages<C, L, NSEQ, THREADS, NS * R, NBUF, INV, SEQ>(v, bufs, par, tw);
        }
    }
}

// Transform of the P0-held data of every thread's sequence (see above). Every
// thread of the CTA calls it. bufs: NBUF buffers of spad_size(NSEQ L) elements.
// With NBUF = 1 the caller must make sure that no thread still reads the
// buffer from an earlier use when this call starts writing it.
template <typename C, int L, int NSEQ, int THREADS, int NBUF, bool INV, int SEQ = spad<C>(L)>
__device__ __forceinline__ void fft_regs(C (&v)[8], C *bufs, int &par, const C *__restrict__ tw)
{
    rfft_stages<C, L, NSEQ, THREADS, 1, NBUF, INV, SEQ>(v, bufs, par, tw);
}
