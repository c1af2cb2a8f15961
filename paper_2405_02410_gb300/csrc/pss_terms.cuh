// pss_terms.cuh -- the explicit terms of FP32 1D and 2D systems with product
// terms, M(q) F[prod_k psi_k^n_k] (arXiv:2405.02410, section "Writing models"),
// in one row kernel for all fields and terms of an instance.
//
// Launched factor by factor, a coupled pair of fields takes 19 launches a step:
// each factor of each term goes back along y and x on its own, through real
// arrays in global memory, and each target forward again.  k_row_terms takes a
// pair of rows of every distinct factor back along x once (plain fields and x
// derivatives from the column kernel's own y inverse; a y derivative or a
// Laplacian from one more y inverse each), keeps the real rows in shared memory,
// evaluates all terms there and transforms one sum per target field.  us per
// step before -> after: a coupled pair at 256^2 92 -> 20 (19 launches -> 2), KPZ at
// 512 x 256 38 -> 18, at 64^2 34 -> 17 (7 -> 3); bound by the chain of one
// pair of rows through its transforms.  2D rows of 16..256 points run on k3_terms
// (pss_regs.cuh); this kernel serves 1D systems and the other lengths.
#pragma once

#include "pss_kernels.cuh"

namespace pss {

template <int N> __host__ __device__ constexpr size_t terms_smem_bytes(int G, int nfac) {
    return sizeof(float2) * ((size_t)(N >= 16 ? N : 0) + (size_t)G * (2 * sf_row(N) + (size_t)nfac * N));
}

template <int N>
__global__ void __launch_bounds__(256) k_row_terms(const TermArgs a) {
    using T = float;
    using C = float2;
    constexpr int EMAX = 8, TPF = FftShape<N, EMAX>::TPF, SF = sf_row(N);
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const SysP<T> &sp = a.sp;
    const TermProg &pg = a.prog;
    const int G = a.G, t = threadIdx.x, nthr = blockDim.x;
    C *TW = reinterpret_cast<C *>(smem_raw);
    C *B0 = TW + twiddle_elems<N>();
    C *B1 = B0 + G * SF;
    C *R = B1 + G * SF;                                       // [pair][factor][x]: the real rows a + i b
    const int inst = blockIdx.y, slot0 = inst * a.nf;
    const int rows = sp.rows, r0 = blockIdx.x * 2 * G;
    const int g = t / TPF, lane = t - g * TPF;
    const bool active = g < G;
    for (int i = t; i < twiddle_elems<N>(); i += nthr) TW[i] = a.tw[twiddle_offset(N, EMAX) + i];
    __syncthreads();
    pdl_wait();
    pdl_trigger();
    const int ra = r0 + 2 * g, rb = ra + 1;                   // this group's rows (1D: the second one is empty)
    const bool has_a = active && ra < rows, has_b = active && rb < rows;
    C *b0 = B0 + (active ? g : 0) * SF, *b1 = B1 + (active ? g : 0) * SF;
    C *Rg = R + (size_t)(active ? g : 0) * pg.nfac * N;
    // ---- every factor's rows to real space
#pragma unroll 1
    for (int f = 0; f < pg.nfac; ++f) {
        const TermFactor fc = pg.fac[f];
        const int slot = slot0 + fc.field;
        const C *__restrict__ in = (fc.arr < 0 ? a.in : a.extra + (size_t)fc.arr * a.extra_stride) +
                                   (size_t)slot * a.slot_stride;
        const int kxc = a.fps[slot].kx_cols;
        fft_run<T, N, EMAX, +1>(
            [&](int k) {
                const int kk = k <= N / 2 ? k : N - k;
                C xa = mk<T>(0, 0), xb = mk<T>(0, 0);
                if (kk < kxc) {
                    const C *p = in + ((size_t)(kk >> 2) * rows + ra) * W + (kk & 3);
                    if (has_a) xa = __ldcg(p);
                    if (has_b) xb = __ldcg(p + W);
                }
                if (fc.dx) {                                  // times i q_x, 0 at the Nyquist index
                    const T q = 2 * kk == N ? T(0) : T(kk) * sp.gx;
                    xa = mk<T>(-q * xa.y, q * xa.x);
                    xb = mk<T>(-q * xb.y, q * xb.x);
                }
                if (k > N / 2) { xa.y = -xa.y; xb.y = -xb.y; }
                if (k == 0 || 2 * k == N) { xa.y = T(0); xb.y = T(0); }
                return mk<T>(xa.x - xb.y, xa.y + xb.x);
            },
            [&](int p, C v, C *) { Rg[f * N + p] = v; }, b0, b1, lane, active, TW);
        __syncthreads();
    }
    // ---- per target field: the sum of its terms, forward along x
#pragma unroll 1
    for (int f = 0; f < a.nf; ++f) {
        if (pg.nterm[f] == 0) continue;
        const int slot = slot0 + f;
        const T *coef = a.coef + (size_t)slot * kMaxTerms;
        const int which = fft_run<T, N, EMAX, -1>(
            [&](int x) {
                C u = mk<T>(0, 0);
                for (int i = 0; i < pg.nterm[f]; ++i) {
                    const TermP &tm = pg.term[f][i];
                    T pa = coef[i], pb = pa;
                    for (int k = 0; k < tm.n; ++k) {
                        const C r = Rg[tm.fac[k] * N + x];
                        for (int e = 0; e < tm.power[k]; ++e) { pa *= r.x; pb *= r.y; }
                    }
                    u.x += pa;
                    u.y += pb;
                }
                return u;
            },
            [&](int p, C v, C *fr) { fr[spad(p)] = v; }, b0, b1, lane, active, TW);
        __syncthreads();
        const C *Z = which == 0 ? B0 : B1;
        C *__restrict__ dst = a.out + (size_t)slot * a.slot_stride;
#pragma unroll 1
        for (int i = t; i < sp.ntiles * 2 * G * W; i += nthr) {
            const int cc = i & 3, rl = (i >> 2) % (2 * G), tl = (i >> 2) / (2 * G);
            if (r0 + rl >= rows) continue;
            const int kx = tl * W + cc;
            C val = mk<T>(0, 0);
            if (kx <= N / 2) {
                const C *z = Z + (rl >> 1) * SF;
                const C wk = z[spad(kx)], wm = z[spad((N - kx) & (N - 1))];
                val = (rl & 1) ? mk<T>(T(0.5) * (wk.y + wm.y), T(-0.5) * (wk.x - wm.x))
                               : mk<T>(T(0.5) * (wk.x + wm.x), T(0.5) * (wk.y - wm.y));
            }
            dst[((size_t)tl * rows + r0 + rl) * W + cc] = val;
        }
        __syncthreads();
    }
    if (a.inc_step && blockIdx.x == 0 && blockIdx.y == 0 && t == 0) *a.d_step += 1;
}

template <int N> cudaError_t launch_terms_n(const TermArgs &a, int batch, cudaStream_t st) {
    constexpr int TPF = FftShape<N, 8>::TPF;
    const int threads = a.G * TPF < 32 ? 32 : a.G * TPF;
    const size_t smem = terms_smem_bytes<N>(a.G, a.prog.nfac);
    if (a.G < 1 || threads > 256 || a.prog.nfac < 1 || a.prog.nfac > kMaxTermFactors) return cudaErrorInvalidConfiguration;
    cudaError_t e = ensure_smem(k_row_terms<N>, smem);
    if (e != cudaSuccess) return e;
    return launch_pdl(k_row_terms<N>, dim3((a.sp.rows + 2 * a.G - 1) / (2 * a.G), batch), threads, smem, st, a);
}

}  // namespace pss
