// pss_resident2d.cuh -- the FP32 2D step of small lattices and of ensembles
// with the whole state on chip (arXiv:2405.02410, section "What cuPSS
// calculates", Eq. timeupdate).
//
// One thread-block cluster holds one slot (one field of one instance) for a
// whole run of steps: the half spectrum's columns and the row pairs are split
// over the cluster's C CTAs (C = 1 .. 16), the two transposes of a step go
// through distributed shared memory, and two cluster barriers separate the
// column phase (forward y FFT, update, inverse y FFT) from the row phase (C2R,
// power, R2C).  Nothing but the state at the start and the end of a run
// crosses to global memory, and clusters never wait for each other, so any
// number of instances runs in one launch, as many at a time as fit.
//
// What bounds it, and why this shape.  The two-kernel step of a small lattice
// is a chain of two launches on a handful of CTAs; an ensemble's is bound by
// issue (profiles/k2_col_k2_row_model_b_512x512_batch40_f32.md), a good part
// of it staging and address arithmetic.  Here a transform of N points is two
// register passes (N = E x N / E, E = 8 or 16) by N / E threads of one warp
// with one padded exchange in shared memory: no CTA barriers inside a
// transform, all offsets compile-time constants, both ends of every transform
// chained in registers (product column -> FFT -> update -> FFT -> transpose;
// staged rows -> FFT -> power -> FFT -> split -> transpose).  A full CTA (128^2
// on one CTA, 128 instances on the chip) issues on 67 % of cycles: it is bound
// by its instructions, 37 % of them transforms, 20 % noise.  Few instances are
// split over more CTAs, where the chain of one phase's instructions per thread
// bounds the step; 8 values per thread instead of 16 took the 128^2 step from
// 7.0 to 4.8 us.  Per step, before -> after: 64^2 10.4 -> 3.2 us, 128^2 11.6
// -> 4.1, 64^2 x 128 instances 13.7 -> 4.7, 128^2 x 128 27.3 -> 13.1.
#pragma once

#include "pss_fast2d.cuh"

namespace pss {

// A transform of N points by TPF threads of one warp, E values per thread:
// thread gl holds points gl + TPF m, before and after.  N = 512 splits its
// second pass in 16 x 2, the radix-2 part by lane exchange.
template <int N> struct RShape {
    static_assert(N == 32 || N == 64 || N == 128 || N == 256 || N == 512, "sides of 32..512 points");
    static constexpr int E = res_e(N);
    static constexpr int TPF = N / E;
    static constexpr bool SPLIT = TPF > E;                // second pass of TPF = 2 E points: E x 2
    static_assert(!SPLIT || TPF == 2 * E, "at most two lanes per second-pass transform");
    static constexpr int R2 = SPLIT ? E : TPF;            // second radix
    static constexpr int BPT = E / R2;                    // second-pass butterflies per thread
    static_assert(TPF >= 4 && TPF <= 32, "a transform's threads share a warp");
    static constexpr int XLD = res_xld(N);                // one transform's buffer: E rows of TPF + 1, and 2 (mod 4)
    // In a warp, groups g and g + 1 work on lines 8 / (16 / TPF) apart (a
    // permutation within blocks of 8), so that the half-warps that access
    // shared memory together fall on distinct banks (lines XLD apart).
    __device__ static __forceinline__ int line(int g) {
        if constexpr (TPF >= 16) {
            return g;
        } else {
            constexpr int GH = 16 / TPF;
            const int low = g & 7;
            return (g & ~7) | ((low % GH) * (TPF / 2) + low / GH);
        }
    }
};

// Unnormalised forward FFT (exponent -2 pi i) of x[] in place; buf: the
// group's XLD points of shared memory, free on entry once the warp meets
// (values read from it before the call may still be in flight to registers of
// other lanes); tw[k TPF + gl] = exp(-2 pi i k gl / N).  `on`: the group has a
// line (its buffer may be written).  Every lane of the warp takes part.
template <int N> __device__ __forceinline__ void rfft(float2 (&x)[RShape<N>::E], float2 *buf, int gl, bool on,
                                                      const float2 *__restrict__ tw) {
    using S = RShape<N>;
    constexpr int E = S::E, TPF = S::TPF, R2 = S::R2, BPT = S::BPT;
    dft_reg<E, -1, float>(x);
#pragma unroll
    for (int k = 1; k < E; ++k) x[k] = cmul<float>(x[k], tw[k * TPF + gl]);
    __syncwarp();
    if (on) {
#pragma unroll
        for (int k = 0; k < E; ++k) buf[k * (TPF + 1) + gl] = x[k];
    }
    __syncwarp();
    if constexpr (!S::SPLIT) {
#pragma unroll
        for (int s = 0; s < BPT; ++s) {
            float2 u[R2];
#pragma unroll
            for (int n = 0; n < R2; ++n) u[n] = buf[(gl + TPF * s) * (TPF + 1) + n];
            dft_reg<R2, -1, float>(u);
#pragma unroll
            for (int k = 0; k < R2; ++k) x[s + BPT * k] = u[k];
        }
    } else {
        // 2 E points per k1 = gl mod E: lanes below E the even ones, the others
        // the odd ones; F[k + E h] = E[k] + (-1)^h exp(-2 pi i k / 2E) O[k]
        const int k1 = gl & (E - 1), odd = gl / E;
        float2 u[E];
#pragma unroll
        for (int n = 0; n < E; ++n) u[n] = buf[k1 * (TPF + 1) + 2 * n + odd];
        dft_reg<E, -1, float>(u);
#pragma unroll
        for (int k = 1; k < E; ++k) {
            const float2 r = rot32<-1, float>(u[k], k * (16 / E));
            if (odd) u[k] = r;
        }
        // lane (k1, odd) finishes k = 2 j + odd for both h: points gl + TPF (j + E/2 h)
#pragma unroll
        for (int j = 0; j < E / 2; ++j) {
            const float2 give = odd ? u[2 * j] : u[2 * j + 1];
            const float2 got = mk<float>(__shfl_xor_sync(0xffffffffu, give.x, E),
                                         __shfl_xor_sync(0xffffffffu, give.y, E));
            const float2 e = odd ? got : u[2 * j], o = odd ? u[2 * j + 1] : got;
            x[j] = cadd<float>(e, o);
            x[j + E / 2] = csub<float>(e, o);
        }
    }
}

// A CTA's shared memory (in complex values after the parameters): the roots of
// both transforms, the state columns PHI, the product columns XC, the row
// pairs XR ([pair][k][row of the pair]).
template <int NX, int NY> struct RSmem {
    static constexpr int LDP = NY + 2;                    // a state column
    static constexpr int LDC = RShape<NY>::XLD;           // a product column
    static constexpr int LDR = RShape<NX>::XLD;           // a row pair (NX + 2 values, or one transform)
    static constexpr int UC = (NX / 2 + 2) / 2;           // column pairs 2u, 2u + 1
    __host__ __device__ static int cols(int C) { return 2 * ((UC + C - 1) / C); }
    __host__ __device__ static int pairs(int C) { return NY / 2 / C; }
    __host__ __device__ static size_t bytes(int C) { return res2_smem_bytes(NX, NY, C); }
    // transform threads: every column and every row pair at once where the
    // register file takes it
    __host__ __device__ static int threads(int C) {
        const int a = cols(C) * RShape<NY>::TPF, b = pairs(C) * RShape<NX>::TPF;
        const int t = ((a > b ? a : b) + 31) / 32 * 32;
        return t > kResMaxThreads ? kResMaxThreads : t;
    }
};

__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire;" ::: "memory");
}
__device__ __forceinline__ uint32_t cluster_rank() {
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}
// the address of this CTA's shared address `a` in CTA `rank` of the cluster
__device__ __forceinline__ uint32_t cluster_map(uint32_t a, uint32_t rank) {
    uint32_t r;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(rank));
    return r;
}
__device__ __forceinline__ void cluster_st(uint32_t a, float2 v) {
    asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void cluster_st4(uint32_t a, float2 v, float2 w) {
    asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(w.x), "f"(w.y)
                 : "memory");
}

// lane of the group's thread that holds points -(gl + TPF m) mod N
template <int N> __device__ __forceinline__ int mirror_lane(int gl) {
    const int base = (int)(threadIdx.x & 31) - gl;
    return base + ((RShape<N>::TPF - gl) & (RShape<N>::TPF - 1));
}
__device__ __forceinline__ float2 shfl2(float2 v, int lane) {
    return mk<float>(__shfl_sync(0xffffffffu, v.x, lane), __shfl_sync(0xffffffffu, v.y, lane));
}

template <int NX, int NY>
__global__ void __launch_bounds__(kResMaxThreads + 32 * kResNoiseWarps, 1) k_res2d(const Res2Args a) {
    using C2 = float2;
    using SX = RShape<NX>;
    using SY = RShape<NY>;
    using L = RSmem<NX, NY>;
    constexpr int EX = SX::E, EY = SY::E;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const SysP<float> &sp = a.sp;
    const int C = a.C, logC = __ffs(C) - 1;
    const int rank = C > 1 ? (int)cluster_rank() : 0;
    const int slot = (int)(blockIdx.x >> logC);
    const int ncl = L::cols(C), npl = L::pairs(C), lognpl = __ffs(npl) - 1;
    FieldP<float> &fp = *reinterpret_cast<FieldP<float> *>(smem_raw);
    static_assert(sizeof(FieldP<float>) <= 192, "the parameters fit before the arrays");
    uint32_t &step0 = *reinterpret_cast<uint32_t *>(smem_raw + 192);
    uint32_t *ctr = reinterpret_cast<uint32_t *>(smem_raw + 200);
    C2 *TWX = reinterpret_cast<C2 *>(smem_raw + 256);
    C2 *TWY = TWX + NX;
    C2 *PHI = TWY + NY;
    C2 *XC = PHI + ncl * L::LDP;
    C2 *XR = XC + ncl * L::LDC;
    const int t = threadIdx.x, nthr = blockDim.x;
    const int nt = nthr - 32 * kResNoiseWarps;           // transform threads, then the noise warps
    auto sync_all = [&]() {
        if (C == 1) __syncthreads();
        else cluster_sync();
    };
    // local column c holds kx = 2 ((c / 2) C + rank) + (c & 1): column pairs go
    // round the CTAs in turn, so that the kept columns (which also transform
    // back) are spread evenly
    auto col_kx = [&](int c) { return 2 * (((c >> 1) << logC) + rank) + (c & 1); };

    // ---- set-up: roots, parameters, the state
    for (int i = t; i < NX; i += nthr)
        TWX[i] = a.roots[((i / SX::TPF) * (i % SX::TPF)) * (kMaxFftN / NX)];
    for (int i = t; i < NY; i += nthr)
        TWY[i] = a.roots[((i / SY::TPF) * (i % SY::TPF)) * (kMaxFftN / NY)];
    for (int i = t; i < (int)(sizeof(FieldP<float>) / 4); i += nthr)
        reinterpret_cast<uint32_t *>(&fp)[i] = reinterpret_cast<const uint32_t *>(&a.fps[slot])[i];
    if (t == 0) {
        step0 = (uint32_t)(*a.d_step);
        ctr[0] = ctr[1] = 0u;
    }
    C2 *__restrict__ gstate = a.state + (size_t)slot * a.slot_stride;
    auto gpos = [&](int kx0, int y) { return ((size_t)(kx0 >> 2) * NY + y) * kTileW + (kx0 & 3); };
    for (int i = t; i < (ncl / 2) * NY; i += nthr) {
        const int u = i / NY, y = i - u * NY, kx0 = col_kx(2 * u);
        C2 v = mk<float>(0.f, 0.f), w = v;
        if (kx0 < sp.hx) ld_pair<float>(gstate + gpos(kx0, y), v, w);
        PHI[(2 * u) * L::LDP + y] = v;
        PHI[(2 * u + 1) * L::LDP + y] = w;
    }
    sync_all();   // also: every CTA of the cluster has started, its shared memory may be written
    const int kmx = fp.kmax[0], kmy = fp.kmax[1], power = fp.power;
    const bool has_product = power > 0;
    const float scale = sp.inv_nsites;
    const uint32_t xr0 = smem_u32(XR), xc0 = smem_u32(XC);

    // ---- the next update's noise, added to the state columns while the row
    // phase runs (Eq. timeupdate adds it to phi_q): 64 pairs of modes at a time,
    // taken from a counter by every warp that has nothing else to do, the noise
    // warps from the start and each transform warp once its rows are done.
    // (Four warps alone made the 128^2 step on one CTA 24 us, twice its
    // transforms; shared out, 15 us, and 13 with the cheaper draws of noise_mode.)
    auto draw_noise = [&](int n) {
        if (!fp.noisy) return;
        const uint32_t step = step0 + (uint32_t)n;
        const float sigma0 = fp.sigma0;
        const int npow = fp.noise_pow, items = (ncl / 2) * NY;
        const PhiloxKey key = philox_key(fp.seed_lo, fp.seed_hi);
        for (;;) {
            int i0 = 0;
            if ((t & 31) == 0) i0 = (int)atomicAdd(&ctr[n & 1], 64u);
            i0 = __shfl_sync(0xffffffffu, i0, 0);
            if (i0 >= items) return;
#pragma unroll
            for (int w = 0; w < 2; ++w) {
                const int i = i0 + 32 * w + (t & 31);
                const int u = i / NY, y = i - u * NY, kx0 = col_kx(2 * u);
                if (i < items && kx0 < sp.hx) {
                    const float qy = fmul(float(signed_k(y, NY)), sp.gy);
                    const float qx0 = fmul(float(kx0), sp.gx), qx1 = fmul(float(kx0 + 1), sp.gx);
                    C2 n0 = mk<float>(0.f, 0.f), n1 = n0;
                    noise_pair<float>(kx0 == 0 || 2 * kx0 == NX, kx0, y, 0,
                                      sigma0, npow, q2sum(qx0, qy), q2sum(qx1, qy), kx0 + 1 < sp.hx, sp,
                                      (uint32_t)fp.field_id, key, step, n0, n1);
                    C2 *p0 = PHI + (2 * u) * L::LDP + y, *p1 = p0 + L::LDP;
                    const C2 f0 = *p0, f1 = *p1;
                    *p0 = mk<float>(fadd(f0.x, n0.x), fadd(f0.y, n0.y));
                    *p1 = mk<float>(fadd(f1.x, n1.x), fadd(f1.y, n1.y));
                }
            }
        }
    };

    if (t >= nt) {
        sync_all();                              // the start's inverse transforms
        for (int n = 0; n < a.nsteps; ++n) {
            draw_noise(n);
            sync_all();                          // row phase done
            if (t == nt) ctr[n & 1] = 0u;                // for step n + 2 (step n + 1 uses the other)
            sync_all();                          // column phase done
        }
    } else {
        float dtO[kPolyTerms], dtM[kPolyTerms];
#pragma unroll
        for (int i = 0; i < kPolyTerms; ++i) {
            dtO[i] = sp.dt * fp.O[i];
            dtM[i] = sp.dt * fp.M[i];
        }
        const bool low = dtO[3] == 0.f && dtO[4] == 0.f && dtM[3] == 0.f && dtM[4] == 0.f;
        // ---- column phase.  first: no product yet, only the inverse transforms
        // of the state; last: no inverse transforms
        auto col_phase = [&](bool first, bool last) {
            const int gl = t & (SY::TPF - 1), ng = nt / SY::TPF;
            const int mir = mirror_lane<NY>(gl);
#pragma unroll 1
            for (int g = t / SY::TPF; (g & ~7) < ncl; g += ng) {
                const int c = SY::line(g), kx = col_kx(c);
                const bool on = c < ncl && kx < sp.hx;
                if (!__any_sync(0xffffffffu, on)) continue;
                C2 *col = XC + (on ? c : 0) * L::LDC;
                C2 *phi = PHI + (on ? c : 0) * L::LDP + gl;
                C2 x[EY];
                if (!first) {
                    if (has_product) {
#pragma unroll
                        for (int m = 0; m < EY; ++m) x[m] = col[gl + SY::TPF * m];
                        rfft<NY>(x, col, gl, on, TWY);
                    }
                    // Eq. timeupdate (the noise is in phi already): g (phi + m P)
                    const float qx = fmul(float(kx), sp.gx);
                    auto update = [&](auto factors) {
#pragma unroll
                        for (int m = 0; m < EY; ++m) {
                            const int ks = gl + SY::TPF * m - (m < EY / 2 ? 0 : NY);
                            const float qy = fmul(float(ks), sp.gy);
                            float fm, fg;
                            factors(q2sum(qx, qy), fm, fg);
                            C2 v = phi[SY::TPF * m];
                            if (has_product) v = mk<float>(ffma(fm, x[m].x, v.x), ffma(fm, x[m].y, v.y));
                            x[m] = cscale<float>(v, fg);
                        }
                    };
                    // operators of degree 2 in q^2 (Models A and B) take the short polynomials
                    if (low)
                        update([&](float q2, float &fm, float &fg) {
                            fm = ffma(ffma(dtM[2], q2, dtM[1]), q2, dtM[0]);
                            fg = fast_rcp(fadd(1.f, ffma(ffma(dtO[2], q2, dtO[1]), q2, dtO[0])));
                        });
                    else
                        update([&](float q2, float &fm, float &fg) { update_factors<float>(q2, dtO, dtM, fm, fg); });
                    // Hermitian part on the kx = 0, Nx/2 columns: with the value at -ky
                    const bool plane = on && (kx == 0 || 2 * kx == NX);
                    if (__any_sync(0xffffffffu, plane)) {
                        if (plane && gl == 0) {
                            x[0].y = 0.f;
                            x[EY / 2].y = 0.f;
#pragma unroll
                            for (int m = 1; m < EY / 2; ++m) {
                                const C2 h = mk<float>(0.5f * (x[m].x + x[EY - m].x), 0.5f * (x[m].y - x[EY - m].y));
                                x[m] = h;
                                x[EY - m] = mk<float>(h.x, -h.y);
                            }
                        }
#pragma unroll
                        for (int m = 0; m < EY / 2; ++m) {
                            const C2 pa = shfl2(x[m], mir), pb = shfl2(x[EY - 1 - m], mir);
                            if (plane && gl != 0) {
                                x[m] = mk<float>(0.5f * (x[m].x + pb.x), 0.5f * (x[m].y - pb.y));
                                x[EY - 1 - m] = mk<float>(0.5f * (x[EY - 1 - m].x + pa.x), 0.5f * (x[EY - 1 - m].y - pa.y));
                            }
                        }
                    }
                    if (on) {
#pragma unroll
                        for (int m = 0; m < EY; ++m) phi[SY::TPF * m] = x[m];
                    }
                } else {
#pragma unroll
                    for (int m = 0; m < EY; ++m) x[m] = phi[SY::TPF * m];
                }
                const bool kept = on && kx <= kmx && has_product;
                if (last || !__any_sync(0xffffffffu, kept)) continue;
                // conjugate of the y inverse of the de-aliased, 1/N-scaled column,
                // to the row pairs' owners
#pragma unroll
                for (int m = 0; m < EY; ++m) {
                    const int ks = gl + SY::TPF * m - (m < EY / 2 ? 0 : NY);
                    const float s = (kept && abs(ks) <= kmy) ? scale : 0.f;
                    x[m] = mk<float>(fmul(x[m].x, s), -fmul(x[m].y, s));
                }
                rfft<NY>(x, col, gl, on, TWY);
                if (kept) {
#pragma unroll
                    for (int m = 0; m < EY; ++m) {
                        const int y = gl + SY::TPF * m, pr = y >> 1;
                        const int ofs = (pr & (npl - 1)) * L::LDR + 2 * kx + (y & 1);
                        if (C == 1) XR[ofs] = x[m];
                        else cluster_st(cluster_map(xr0 + 8u * (uint32_t)ofs, (uint32_t)(pr >> lognpl)), x[m]);
                    }
                }
            }
        };
        // ---- row phase: two rows per transform (z = a + i b), as k2_row
        auto row_phase = [&]() {
            const int gl = t & (SX::TPF - 1), ng = nt / SX::TPF;
            const int mir = mirror_lane<NX>(gl);
#pragma unroll 1
            for (int g = t / SX::TPF; (g & ~7) < npl; g += ng) {
                const int j = SX::line(g);
                const bool on = j < npl;
                if (!__any_sync(0xffffffffu, on)) continue;
                C2 *row = XR + (on ? j : 0) * L::LDR;
                C2 x[EX];
                // Y = conj(Z) from the stored conjugates at column k: Y_k here,
                // Y_{N-k} for the lane that holds point N - k
                C2 yh = mk<float>(0.f, 0.f);
                if (gl == 0 && kmx >= NX / 2) {
                    const float4 ab = *reinterpret_cast<const float4 *>(row + NX);
                    yh = mk<float>(ab.x, -ab.z);
                }
                C2 z0 = mk<float>(0.f, 0.f);             // lane 0's value for its point E - m
#pragma unroll
                for (int m = EX / 2 - 1; m >= 0; --m) {
                    const int k = gl + SX::TPF * m;
                    float4 ab = make_float4(0.f, 0.f, 0.f, 0.f);
                    if (k <= kmx) ab = *reinterpret_cast<const float4 *>(row + 2 * k);
                    if (m == 0 && gl == 0) { ab.y = 0.f; ab.w = 0.f; }
                    x[m] = mk<float>(ab.x + ab.w, ab.y - ab.z);
                    const C2 z = mk<float>(ab.x - ab.w, -ab.y - ab.z);
                    const C2 got = shfl2(z, mir);
                    x[EX - 1 - m] = gl != 0 ? got : (m == EX / 2 - 1 ? yh : z0);
                    z0 = z;
                }
                rfft<NX>(x, row, gl, on, TWX);
                // z' = conj(z) = a - i b; u = a^p + i b^p
#pragma unroll
                for (int m = 0; m < EX; ++m) {
                    const float p = x[m].x, q = -x[m].y;
                    if (power == 3) x[m] = mk<float>(fmul(fmul(p, p), p), fmul(fmul(q, q), q));
                    else if (power == 2) x[m] = mk<float>(fmul(p, p), fmul(q, q));
                    else x[m] = mk<float>(p, q);
                }
                rfft<NX>(x, row, gl, on, TWX);
                // the two rows' half spectra to the columns' owners: rows 2 j', 2 j' + 1
                // of column k are 16 bytes
                const int y0 = 2 * ((rank << lognpl) + j);
                auto push = [&](int k, C2 wk, C2 wm) {
                    const int u = k >> 1;
                    const int ofs = (2 * (u >> logC) + (k & 1)) * L::LDC + y0;
                    const C2 A = mk<float>(0.5f * (wk.x + wm.x), 0.5f * (wk.y - wm.y));
                    const C2 B = mk<float>(0.5f * (wk.y + wm.y), -0.5f * (wk.x - wm.x));
                    if (C == 1) st_pair<float>(XC + ofs, A, B);
                    else cluster_st4(cluster_map(xc0 + 8u * (uint32_t)ofs, (uint32_t)(u & (C - 1))), A, B);
                };
#pragma unroll
                for (int m = 0; m < EX / 2; ++m) {
                    const C2 got = shfl2(x[EX - 1 - m], mir);
                    const C2 wm = gl != 0 ? got : x[m == 0 ? 0 : EX - m];
                    if (on) push(gl + SX::TPF * m, x[m], wm);
                }
                if (on && gl == 0) push(NX / 2, x[EX / 2], x[EX / 2]);
            }
        };
        if (has_product) col_phase(true, false);
        sync_all();
        for (int n = 0; n < a.nsteps; ++n) {
            if (has_product) row_phase();
            draw_noise(n);
            sync_all();
            col_phase(false, n + 1 == a.nsteps);
            sync_all();
        }
    }
    bool bad = false;
    // ---- the state goes back; the last slot to finish advances the step counter
    for (int i = t; i < (ncl / 2) * NY; i += nthr) {
        const int u = i / NY, y = i - u * NY, kx0 = col_kx(2 * u);
        if (kx0 < sp.hx) {
            const C2 v = PHI[(2 * u) * L::LDP + y];
            const C2 w = kx0 + 1 < sp.hx ? PHI[(2 * u + 1) * L::LDP + y] : mk<float>(0.f, 0.f);
            st_pair<float>(gstate + gpos(kx0, y), v, w);
            // a mode that became NaN or infinite stays so: one check at the end
            bad |= !(fabsf(v.x) + fabsf(v.y) + fabsf(w.x) + fabsf(w.y) <= 3.0e38f);
        }
    }
    if (bad && a.d_status) atomicOr(a.d_status, kStatusNonFinite);
    if (t == 0) {
        __threadfence();
        if (atomicAdd(&a.gs->done, 1u) + 1u == gridDim.x) {
            a.gs->done = 0u;
            *a.d_step += a.nsteps;   // every CTA has read it
        }
    }
}

// active != nullptr: only how many clusters of C CTAs run at a time
template <int NX, int NY> cudaError_t launch_res2_n(const Res2Args &a, int nslots, cudaStream_t st, int *active) {
    using L = RSmem<NX, NY>;
    const int C = a.C;
    const size_t smem = L::bytes(C);
    if (C < 1 || C > 16 || (C & (C - 1)) || L::pairs(C) < 1 || smem > 227 * 1024) return cudaErrorInvalidConfiguration;
    cudaError_t e = ensure_smem(k_res2d<NX, NY>, smem);
    if (e == cudaSuccess && C > 8)
        e = cudaFuncSetAttribute(k_res2d<NX, NY>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(nslots * C, 1, 1);
    cfg.blockDim = dim3(L::threads(C) + 32 * kResNoiseWarps, 1, 1);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = C;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (active) return cudaOccupancyMaxActiveClusters(active, k_res2d<NX, NY>, &cfg);
    return cudaLaunchKernelEx(&cfg, k_res2d<NX, NY>, a);
}

template <int NX> cudaError_t launch_res2_nx(const Res2Args &a, int nslots, cudaStream_t st, int *active) {
    switch (a.sp.ny) {
        case 32: return launch_res2_n<NX, 32>(a, nslots, st, active);
        case 64: return launch_res2_n<NX, 64>(a, nslots, st, active);
        case 128: return launch_res2_n<NX, 128>(a, nslots, st, active);
        case 256: return launch_res2_n<NX, 256>(a, nslots, st, active);
        case 512: return launch_res2_n<NX, 512>(a, nslots, st, active);
        default: return cudaErrorInvalidValue;
    }
}

}  // namespace pss
