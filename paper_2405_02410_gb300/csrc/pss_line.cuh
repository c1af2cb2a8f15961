// pss_line.cuh -- a run of steps of a 1D lattice in one launch, one CTA per
// slot (arXiv:2405.02410, section "What cuPSS calculates", Eq. timeupdate).
//
// A line of up to 1024 sites is a few kilobytes: its steps are bound by the
// latency of launches and of one transform's passes, and in FP64 by the one
// SM's arithmetic.  The state, the product and the transform buffers stay in
// shared memory for the whole run; a real transform of N points is a complex
// one of N / 2 (even sites in the real, odd ones in the imaginary part), half
// the work of the row kernel's pair transform with an empty second row; the
// untangling rides on the update's reads and, in FP32, on the first pass's
// loads.  FP32 takes radix 4 (fewest cycles per pass times passes at one warp
// per scheduler).  FP64 takes radix 2 with one output per thread, four fused
// multiply-adds each: an FP64 warp instruction takes its scheduler 64 cycles
// however long the others wait, so the passes are spread over all four.  The
// update's factors are tabulated once per launch.  A boundary frame (section
// "Callback functions") is set inside the inverse transform's last pass.
// us per step, the generic kernels' launches -> here: FP32 Model B of 1024
// sites 12.4 -> 2.5, of 64 9.5 -> 1.5; FP64 of 1024 46 -> 28 (one SM's FP64
// units), the framed diffusion of 256 sites in FP64 92 -> 6 (nine launches a
// step, two of them transforms of a product it does not have).
#pragma once

#include "pss_kernels.cuh"

namespace pss {

template <typename T, int N> struct LineShape {
    static constexpr int M = N / 2;
    static constexpr bool WIDE = sizeof(T) == 8;             // one point per thread
    static constexpr int EMAX = WIDE ? 2 : 4;
    static constexpr int TPF = WIDE ? M : FftShape<M, EMAX>::TPF;
    // threads: FP32 one pair of modes each; FP64 one mode each, and a warp for mode M
    static constexpr int NT = WIDE ? M + 32 : M / 2 < 64 ? 64 : M / 2;
    static constexpr int BUF = padded(M);
    static_assert(TPF <= NT, "every transform thread exists");
    // roots of the transform (M) and of the untangling (N: M + 1), the state, the
    // update's factors (M + 1 each, rounded up to even) and two buffers
    static constexpr size_t BYTES = sizeof(cplx<T>) * (size_t)(M + 3 * (M + 2) + 2 * BUF);
};

template <typename T, int N>
__global__ void __launch_bounds__(LineShape<T, N>::NT) k_line(const LineArgs<T> a) {
    using C = cplx<T>;
    using S = LineShape<T, N>;
    constexpr int M = S::M, EMAX = S::EMAX;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ FieldP<T> fp;
    __shared__ uint32_t s_step0;
    C *TW = reinterpret_cast<C *>(smem_raw);
    C *WN = TW + M;
    C *PHI = WN + M + 2;
    C *MG = PHI + M + 2;                                      // dt M(q), 1 / (1 + dt O(q))
    C *B0 = MG + M + 2;
    C *B1 = B0 + S::BUF;
    const SysP<T> &sp = a.sp;
    const int t = threadIdx.x, slot = blockIdx.x;
    const LineField<T> fl = a.fld[slot % a.nf];
    C *__restrict__ gstate = a.state + (size_t)slot * a.slot_stride;
    for (int i = t; i < M; i += S::NT) TW[i] = a.tw[twiddle_offset(M, EMAX) + i];
    for (int i = t; i <= M; i += S::NT) {
        WN[i] = a.tw[kRootsOffset + i * (kMaxFftN / N)];
        PHI[i] = gstate[i];
    }
    for (int i = t; i < (int)(sizeof(FieldP<T>) / 4); i += S::NT)
        reinterpret_cast<uint32_t *>(&fp)[i] = reinterpret_cast<const uint32_t *>(&a.fps[slot])[i];
    if (t == 0) s_step0 = (uint32_t)(*a.d_step);
    __syncthreads();
    const bool active = t < S::TPF;
    const bool has_product = fl.power > 0, noisy = fp.noisy != 0;
    const int kmx = fp.kmax[0], npow = fp.noise_pow;
    const T sigma0 = fp.sigma0;
    {
        T dtO[kPolyTerms], dtM[kPolyTerms];
#pragma unroll
        for (int i = 0; i < kPolyTerms; ++i) {
            dtO[i] = sp.dt * fp.O[i];
            dtM[i] = sp.dt * fp.M[i];
        }
        for (int k = t; k <= M; k += S::NT) {
            const T q = T(k) * sp.gx;
            update_factors<T>(q * q, dtO, dtM, MG[k].x, MG[k].y);
        }
    }
    __syncthreads();   // the update reads factors of other threads, without a product before any other barrier
    const PhiloxKey key = philox_key(fp.seed_lo, fp.seed_hi);

    // Point k of the half-length inverse transform of a half spectrum X:
    // (X_k + conj X_{M-k}) + i exp(2 pi i k / N) (X_k - conj X_{M-k})
    auto tangle = [&](C x, C y, int k) {
        const C s = mk<T>(x.x + y.x, x.y - y.y), d = mk<T>(x.x - y.x, x.y + y.y), w = WN[k];   // w = (cos, -sin)
        // i (w.x - i w.y) d = (w.y + i w.x) d
        return mk<T>(s.x + (w.y * d.x - w.x * d.y), s.y + (w.y * d.y + w.x * d.x));
    };
    // Twice mode k of the half spectrum from the half-length forward transform Z:
    // (Z_k + conj Z_{M-k}) - i exp(-2 pi i k / N) (Z_k - conj Z_{M-k})
    auto untangle2 = [&](const C *Z, int k) {
        const int p = k & (M - 1), r = (M - k) & (M - 1);
        const C x = Z[S::WIDE ? p : spad(p)], y = Z[S::WIDE ? r : spad(r)], w = WN[k];
        const C s = mk<T>(x.x + y.x, x.y - y.y), d = mk<T>(x.x - y.x, x.y + y.y);
        // -i (w.x + i w.y) d = (w.y - i w.x) d
        return mk<T>(s.x + (w.y * d.x + w.x * d.y), s.y + (w.y * d.y - w.x * d.x));
    };
    auto untangle = [&](const C *Z, int k) { return cscale<T>(untangle2(Z, k), T(0.5)); };
    // the real rows of the inverse transform, two sites per complex value, go
    // through `site(n, x)` and forward again; returns the buffer of the result
    auto there_and_back = [&](auto src, auto site) {
        if constexpr (S::WIDE) {
            // points first, then radix-2 passes, thread t the output of sign t mod 2
            // of butterfly t / 2: a +- w b
            C *cur = B0, *nxt = B1;
            if (t < M) cur[t] = src(t);
            __syncthreads();
            const int i = t >> 1;
            auto passes = [&](bool inverse) {
#pragma unroll 1
                for (int P = 1; P < M; P <<= 1) {
                    if (t < M) {
                        const int k = i & (P - 1);
                        const C x = cur[i], y = cur[i + M / 2];
                        C v;
                        if (P == 1) {
                            v = (t & 1) ? csub<T>(x, y) : cadd<T>(x, y);
                        } else {
                            C w = TW[P - 2 + k];
                            if (inverse) w.y = -w.y;
                            if (t & 1) w = mk<T>(-w.x, -w.y);
                            v = mk<T>(ffma(w.x, y.x, ffma(-w.y, y.y, x.x)), ffma(w.x, y.y, ffma(w.y, y.x, x.y)));
                        }
                        if (inverse && 2 * P == M) {
                            const int n = 2 * (k + (t & 1) * P);   // the last pass: butterfly k = i
                            v = mk<T>(site(n, v.x), site(n + 1, v.y));
                        }
                        nxt[((i - k) << 1) + k + (t & 1) * P] = v;
                    }
                    __syncthreads();
                    C *tmp = cur;
                    cur = nxt;
                    nxt = tmp;
                }
            };
            passes(true);
            passes(false);
            return cur;
        } else {
        const int which = fft_run<T, M, EMAX, +1>(
            src, [&](int p, C v, C *fr) { fr[spad(p)] = mk<T>(site(2 * p, v.x), site(2 * p + 1, v.y)); }, B0, B1, t,
            active, TW);
        __syncthreads();
        C *zf = which == 0 ? B0 : B1, *other = which == 0 ? B1 : B0;
        const int which2 = fft_run<T, M, EMAX, -1>([&](int k) { return zf[spad(k)]; },
                                                   [&](int p, C v, C *fr) { fr[spad(p)] = v; }, other, zf, t, active, TW);
        __syncthreads();
        return which2 == 0 ? other : zf;
        }
    };
    // the product of the state: F[(F^-1[op m phi])^power]
    auto product = [&]() {
        auto masked = [&](int k) {
            if (k > kmx) return mk<T>(T(0), T(0));
            C v = cscale<T>(PHI[k], sp.inv_nsites);
            if (k == 0 || k == M) v.y = T(0);
            if (fl.deriv >= 0 || fl.lap > 0) {
                const T q = T(k) * sp.gx;
                T f = T(1);
                for (int l = 0; l < fl.lap; ++l) f *= -(q * q);
                if (fl.deriv >= 0) {
                    const T qf = k == M ? T(0) : q * f;
                    v = mk<T>(-qf * v.y, qf * v.x);
                } else {
                    v = cscale<T>(v, f);
                }
            }
            return v;
        };
        return there_and_back([&](int k) { return tangle(masked(k), masked(M - k), k); },
                              [&](int, T x) { return fl.power == 3 ? x * x * x : ipow<T>(x, fl.power); });
    };

    const C *P = has_product ? product() : nullptr;
    for (int n = 0; n < a.nsteps; ++n) {
        // ---- update (Eq. timeupdate)
        auto update = [&](int k, C xi) {
            const C mg = MG[k];
            C v = update_pre<T>(PHI[k], has_product ? untangle(P, k) : mk<T>(0, 0), xi, mg.x, mg.y, has_product);
            if (k == 0 || k == M) v.y = T(0);           // the field is real
            PHI[k] = v;
        };
        const uint32_t step = s_step0 + (uint32_t)n;
        if constexpr (S::WIDE) {
            if (t <= M) {
                const T q = T(t) * sp.gx;
                C xi = mk<T>(0, 0);
                if (noisy)
                    xi = noise_one<T>(t == 0 || t == M, t, 0, 0, sigma0, npow, q * q, sp, (uint32_t)fp.field_id, key, step,
                                      a.tw);
                update(t, xi);
            }
        } else {
            // modes 2 j and 2 j + 1 per thread: they share a draw
            for (int kx0 = 2 * t; kx0 <= M; kx0 += 2 * S::NT) {
                const T q0 = T(kx0) * sp.gx, q1 = T(kx0 + 1) * sp.gx;
                C x0 = mk<T>(0, 0), x1 = x0;
                if (noisy)
                    noise_pair<T>(kx0 == 0 || kx0 == M, kx0, 0, 0, sigma0, npow, q0 * q0, q1 * q1, kx0 < M, sp,
                                  (uint32_t)fp.field_id, key, step, x0, x1, a.tw);
                update(kx0, x0);
                if (kx0 < M) update(kx0 + 1, x1);
            }
        }
        __syncthreads();
        if (fl.frame_w > 0) {
            // the change that sets the frame on the real field, zero inside it, added to
            // the spectrum: the transforms' roundings reach the state by the size of that
            // change, not of the field
            auto full = [&](int k) {
                C v = cscale<T>(PHI[k], sp.inv_nsites);
                if (k == 0 || k == M) v.y = T(0);
                return v;
            };
            const C *Z = there_and_back([&](int k) { return tangle(full(k), full(M - k), k); },
                                        [&](int x, T v) {
                                            const bool lo = x < fl.frame_w;
                                            const T b = lo ? fl.frame_lo : fl.frame_hi;
                                            return lo || x >= N - fl.frame_w ? b - v : T(0);
                                        });
            for (int k = t; k <= M; k += S::NT) {
                const C d = untangle2(Z, k), h = PHI[k];
                PHI[k] = mk<T>(ffma(T(0.5), d.x, h.x), ffma(T(0.5), d.y, h.y));
            }
            __syncthreads();
        }
        if (has_product && n + 1 < a.nsteps) P = product();
    }
    bool bad = false;
    for (int k = t; k <= M; k += S::NT) {
        gstate[k] = PHI[k];
        bad |= !finite_mode(PHI[k]);                     // a mode that became NaN or infinite stays so
    }
    if (bad && a.d_status) atomicOr(a.d_status, kStatusNonFinite);
    if (t == 0) {
        __threadfence();
        if (atomicAdd(&a.gs->done, 1u) + 1u == gridDim.x) {
            a.gs->done = 0u;
            *a.d_step += a.nsteps;                       // every CTA has read it
        }
    }
}

template <typename T, int N> cudaError_t launch_line_n(const LineArgs<T> &a, int nslots, cudaStream_t st) {
    using S = LineShape<T, N>;
    cudaError_t e = ensure_smem(k_line<T, N>, S::BYTES);
    if (e != cudaSuccess) return e;
    k_line<T, N><<<nslots, S::NT, S::BYTES, st>>>(a);
    return cudaGetLastError();
}

template <typename T> cudaError_t launch_line(const LineArgs<T> &a, int nslots, cudaStream_t st) {
    switch (a.sp.nx) {
        case 64: return launch_line_n<T, 64>(a, nslots, st);
        case 128: return launch_line_n<T, 128>(a, nslots, st);
        case 256: return launch_line_n<T, 256>(a, nslots, st);
        case 512: return launch_line_n<T, 512>(a, nslots, st);
        case 1024: return launch_line_n<T, 1024>(a, nslots, st);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace pss
