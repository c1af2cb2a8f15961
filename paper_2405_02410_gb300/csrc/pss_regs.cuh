// pss_regs.cuh -- the passes of FP32 2D and 3D systems with their points in
// registers (arXiv:2405.02410, section "What cuPSS calculates", Eq. timeupdate).
//
// k_col, k_mid and k_row stage their tiles in shared memory and run every phase from
// there; they are bound by instructions and barriers, not by HBM (k_col at
// 256^3: 257 instructions per mode, 73 % issue-active, 35 % of the DRAM
// rate).  Here a thread keeps E points of a transform of N = R1 E points in
// registers: loads come straight from global memory (consecutive threads take
// a tile's columns and neighbouring positions, whole 128-byte lines), a
// transform is two passes with one exchange through shared memory, and the
// forward transform's outputs (positions lane + r R1) are what the inverse
// one's first pass reads, so the update runs in registers between them.  The
// noise is drawn into shared memory while the loads are in flight, a pair of
// columns per Philox call.  us, staged -> here: 256^3, two fields: z pass 153
// -> 104 (466 MB: 4.5 TB/s), y inverse 52 -> 37, y forward 63 -> 52 (270 MB:
// 5.2 TB/s), x pass 104 -> 66 (225 MB: 3.4 TB/s), the step 351 -> 238; whole
// steps of 128^3 (two fields) 58 -> 35, 256 x 256 x 64 54 -> 34, 64^3 (two fields)
// 22.0 -> 10.7, 32^3 20.4 -> 7.8; 2D batches against the FFT-group kernels: 512^2 x 32
// 85 -> 62, 1024^2 x 8 107 -> 67.  The step's column pass takes 5 CTAs per SM and
// 96 registers, the state among them; 6 CTAs and 80 registers with the state
// copied to shared memory asynchronously measured 118 .. 126 us at 256^3 in place
// of 111; tests of planes, kept positions and the noise's power that hold for the
// whole CTA, hoisted out of the per-mode code, took it from 111 to 104.  512 and 1024 points put 32 points on a thread, so there the state
// goes through shared memory with the noise.

#pragma once

#include "pss_kernels.cuh"

namespace pss {

// N = R1 E: R1 threads per transform, E points each; passes of radix R1 (the
// forward transform's first, BPT butterflies per thread) and E
template <int N> struct R3Shape {
    static constexpr int E = N >= 512 ? 32 : N >= 128 ? 16 : N >= 32 ? 8 : 4;
    static constexpr int R1 = N / E;
    static constexpr int BPT = E / R1;
    static constexpr int CHUNK = W * R1;                 // k3_col: threads per chunk (a tile of a pencil)
    static constexpr int BUF = (N + E) * W;              //   its exchange buffer, one pad position per butterfly
    static constexpr int TWN = R1 == E ? N : 2 * N;      // twiddles [r - 1][k] of the radix-E pass, of the radix-R1 one
    static constexpr bool ALIAS = N >= 512;              //   which then takes the state and noise as well
    static constexpr int CTAS = N >= 512 ? 4 : 6;        // CTAs of 128 threads per SM the registers are held to
    static_assert(R1 <= E && CHUNK <= 128, "shape");
};

// twiddles exp(-2 pi i r k / N): of the radix-E pass after R1 points [r - 1][k < R1], and of
// the radix-R1 pass after E points [r - 1][k < E] at twi (the same where R1 = E)
template <int N> __device__ __forceinline__ void r3_twiddles(float2 *TW, const float2 *__restrict__ tw, int t, int nthr) {
    using S = R3Shape<N>;
    for (int i = t; i < N; i += nthr) {
        if constexpr (S::R1 == S::E) {
            TW[i] = tw[twiddle_offset(N, S::E) + i];
        } else {
            TW[i] = tw[kRootsOffset + ((i / S::R1 + 1) % S::E) * (i % S::R1) * (kMaxFftN / N)];
            TW[N + i] = tw[twiddle_offset(N, S::E) + i];
        }
    }
}

// Modes of k3_col: the step, forward only (COL_FWD), inverse only (COL_INV_MASK, COL_INV_FULL)
enum { R3_STEP = 0, R3_FWD = 1, R3_INV = 2 };

// The z pass in 3D, the y pass in 2D.  A CTA takes tiles (in 3D of the pencils
// ky and -ky: a kx = 0 mode and its Hermitian partner are in one CTA), a chunk
// of CHUNK threads for each; thread: column c, lane, chunk.
template <int N, int MODE, int DIM>
__global__ void __launch_bounds__(128, MODE == R3_STEP && N < 512 ? 5 : R3Shape<N>::CTAS) k3_col(const ColArgs<float> a) {
    using S = R3Shape<N>;
    using C = float2;
    constexpr int E = S::E, R1 = S::R1;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ FieldP<float> fp;
    const SysP<float> &sp = a.sp;
    constexpr bool is3 = DIM == 3;
    const int nthr = is3 ? 128 : blockDim.x;
    const int t = threadIdx.x, c = t & (W - 1), lane = (t >> 2) % R1, ch = t / S::CHUNK;
    const int chunks = nthr / S::CHUNK, ctiles = is3 ? chunks >> 1 : chunks;
    C *TW = reinterpret_cast<C *>(smem_raw);
    C *XCH = TW + S::TWN;
    C *XI = S::ALIAS ? XCH : XCH + chunks * S::BUF;              // R3_STEP: the noise (ALIAS: plus the state), [chunk][pos][W]
    constexpr int XS = S::ALIAS ? S::BUF : N * W;
    const int slot = a.slot0 + blockIdx.z;
    const int op = blockIdx.y, opp = (sp.n_outer - op) & (sp.n_outer - 1);
    const bool lone = is3 && op == opp;                          // its own partner: the second chunk is a copy
    const int first_tile = blockIdx.x * ctiles, tile = first_tile + (is3 ? ch >> 1 : ch);
    const int o = is3 && (ch & 1) ? opp : op, kx = tile * W + c;
    // (one tile per CTA: the grid covers them exactly)
    const bool ok = (is3 && 2 * S::CHUNK == 128) || tile < a.n_tiles, writes = ok && !((ch & 1) && lone);
    const size_t ofs = (size_t)slot * a.slot_stride + ((size_t)tile * sp.n_outer + o) * N * W + c;
    C *xb = XCH + ch * S::BUF + c;
    r3_twiddles<N>(TW, a.tw, t, nthr);
    for (int i = t; i < (int)(sizeof(FieldP<float>) / 4); i += nthr)
        reinterpret_cast<uint32_t *>(&fp)[i] = reinterpret_cast<const uint32_t *>(&a.fps[slot])[i];
    __syncthreads();
    const int oy = is3 ? signed_k(o, sp.ny) : 0;                 // ky of the pencil
    const bool full = a.mode == COL_INV_FULL;
    // CTA-uniform: it holds kx = 0 or Nx/2 (and with Nx/2 the columns past the grid)
    const bool planes = first_tile == 0 || (first_tile * W <= sp.nx / 2 && sp.nx / 2 < (first_tile + ctiles) * W);
    auto kept_o = [&](int k) { return !is3 || abs(signed_k(k, sp.ny)) <= fp.kmax[1]; };
    // CTA-uniform: nothing of the inverse is kept
    const bool inverse = MODE != R3_FWD && (full || (first_tile * W <= fp.kmax[0] && kept_o(op)));
    pdl_wait();
    pdl_trigger();
    if (MODE == R3_INV && !inverse) return;
    const bool keep = kx < sp.hx && (full || (kx <= fp.kmax[0] && kept_o(o)));
    const int kmax_pos = full ? N : is3 ? fp.kmax[2] : fp.kmax[1];
    // whether position lane + r R1 is kept: |k| <= kmax_pos, as bounds on the lane
    const int keep_hi = keep ? kmax_pos : -1, keep_lo = keep ? N - kmax_pos : 2 * N;
    auto kept_pos = [&](int r) { return 2 * r < E ? lane <= keep_hi - r * R1 : lane >= keep_lo - r * R1; };
    const float gpos = is3 ? sp.gz : sp.gy;
    C v[E];                                                      // from the forward transform on: positions lane + r R1
    if constexpr (MODE != R3_INV) {
        const C *__restrict__ in = a.in + ofs;
#pragma unroll
        for (int s = 0; s < S::BPT; ++s)
#pragma unroll
            for (int r = 0; r < R1; ++r) v[s * R1 + r] = ok ? in[(lane + s * R1 + r * E) * W] : mk<float>(0, 0);
        // the noise of the chunk, a pair of columns per thread (they share a Philox
        // call); ALIAS: added to the state
        auto noise = [&]() {
            const int u = t % S::CHUNK, cp = u & 1, kx0 = tile * W + 2 * cp;
            const float qx0 = (float)kx0 * sp.gx, qx1 = (float)(kx0 + 1) * sp.gx, qo = (float)oy * sp.gy;
            const float qx0s = qx0 * qx0, qx1s = qx1 * qx1, qo2 = qo * qo;
            const PhiloxKey key = philox_key(fp.seed_lo, fp.seed_hi);
            const uint32_t step = (uint32_t)(*a.d_step), fid = (uint32_t)fp.field_id;
            // (a test of the whole CTA: most hold neither plane)
            const bool on_plane = planes && (kx0 == 0 || 2 * kx0 == sp.nx), has1 = kx0 + 1 < sp.hx, noisy = !S::ALIAS || fp.noisy != 0;
            const int npow = fp.noise_pow;
            const float sigma0 = fp.sigma0;
            const C *st = a.state + ofs - c + 2 * cp;
            C *xi = XI + ch * XS + 2 * cp;
            C n0 = mk<float>(0, 0), n1 = n0;
            if (S::ALIAS && ok) ld_pair<float>(st + (u >> 1) * W, n0, n1);
            auto draw = [&](auto plane, auto odd) {
#pragma unroll 1
                for (int pos = u >> 1; pos < N; pos += 2 * R1) {
                    C x0 = mk<float>(0, 0), x1 = x0;
                    const C f0 = n0, f1 = n1;
                    if (S::ALIAS && ok && pos + 2 * R1 < N) ld_pair<float>(st + (pos + 2 * R1) * W, n0, n1);   // the next one's
                    if (noisy) {
                        const float qp = (float)signed_k(pos, N) * gpos, qyz2 = qp * qp + qo2;
                        noise_pair<float>(decltype(plane)::value && on_plane, kx0, is3 ? o : pos, is3 ? pos : 0, sigma0, decltype(odd)::value ? 1 : npow, qx0s + qyz2, qx1s + qyz2, has1,
                                          sp, fid, key, step, x0, x1);
                    }
                    if (S::ALIAS) {
                        x0 = mk<float>(fadd(f0.x, x0.x), fadd(f0.y, x0.y));
                        x1 = mk<float>(fadd(f1.x, x1.x), fadd(f1.y, x1.y));
                    }
                    st_pair<float>(xi + pos * W, x0, x1);
                }
            };
            // one of the three forms for the whole CTA: no plane and conserved noise of
            // power 1, no plane, any
            if (planes) draw(std::true_type{}, std::false_type{});
            else if (npow == 1) draw(std::false_type{}, std::true_type{});
            else draw(std::false_type{}, std::false_type{});
        };
        if (MODE == R3_STEP && !S::ALIAS && fp.noisy) noise();
#pragma unroll
        for (int s = 0; s < S::BPT; ++s) {
            dft_reg<R1, -1, float>(v + s * R1);
#pragma unroll
            for (int r = 0; r < R1; ++r) xb[((lane + s * R1) * (R1 + 1) + r) * W] = v[s * R1 + r];
        }
        C ph[S::ALIAS ? 1 : E];
        if (MODE == R3_STEP && !S::ALIAS) {
#pragma unroll
            for (int r = 0; r < E; ++r) ph[r] = ok ? a.state[ofs + (lane + r * R1) * W] : mk<float>(0, 0);
        }
        __syncthreads();
#pragma unroll
        for (int r = 0; r < E; ++r) {
            v[r] = xb[(lane + r * (R1 + 1)) * W];
            if (r > 0) v[r] = cmul<float>(v[r], TW[(r - 1) * R1 + lane]);
        }
        if (MODE == R3_STEP && S::ALIAS) {
            __syncthreads();                                     // the exchange buffer is free
            noise();
            __syncthreads();
        }
        dft_reg<E, -1, float>(v);
        if constexpr (MODE == R3_STEP) {
            const bool has_product = fp.power > 0, noisy = fp.noisy != 0;
            const float qx = (float)kx * sp.gx, qo = (float)oy * sp.gy;
            const float qxs = qx * qx, qo2 = qo * qo;
            const C *xi = XI + ch * XS + c;
            float dtO[kPolyTerms], dtM[kPolyTerms];
#pragma unroll
            for (int i = 0; i < kPolyTerms; ++i) {
                dtO[i] = sp.dt * fp.O[i];
                dtM[i] = sp.dt * fp.M[i];
            }
            bool bad = false;
            auto update = [&](auto degree2) {
#pragma unroll
                for (int r = 0; r < E; ++r) {
                    const float qp = (float)(lane + r * R1 - (2 * r >= E ? N : 0)) * gpos;
                    const float q2 = qxs + (qp * qp + qo2);
                    float m, g;
                    if (decltype(degree2)::value) {
                        m = ffma(ffma(dtM[2], q2, dtM[1]), q2, dtM[0]);
                        g = fast_rcp(fadd(1.0f, ffma(ffma(dtO[2], q2, dtO[1]), q2, dtO[0])));
                    } else {
                        update_factors<float>(q2, dtO, dtM, m, g);
                    }
                    // (ALIAS: phi + xi in place of xi; the same sum)
                    const C f = S::ALIAS ? mk<float>(0, 0) : ph[S::ALIAS ? 0 : r];
                    const C x = S::ALIAS || noisy ? xi[(lane + r * R1) * W] : mk<float>(0, 0);
                    v[r] = update_pre<float>(f, v[r], x, m, g, has_product);
                    bad |= !finite_mode(v[r]);
                }
            };
            // operators of degree 2 in q^2 (Models A and B) take the short polynomials
            if (dtO[3] == 0.0f && dtO[4] == 0.0f && dtM[3] == 0.0f && dtM[4] == 0.0f) update(std::true_type{});
            else update(std::false_type{});
            if (bad && ok && kx < sp.hx && a.d_status) atomicOr(a.d_status, kStatusNonFinite);
        }
        // Hermitian part on the kx = 0 and Nx/2 planes (the field is real): phi(k) <-
        // (phi(k) + conj phi(-k)) / 2, the partner at position -pos (of the partner pencil)
        if (planes) {
            const bool plane = ok && (kx == 0 || 2 * kx == sp.nx);
            __syncthreads();
            if (plane) {
#pragma unroll
                for (int r = 0; r < E; ++r) xb[(lane + r * R1) * W] = v[r];
            }
            __syncthreads();
            if (plane) {
                const C *pb = XCH + (is3 ? ch ^ 1 : ch) * S::BUF + c;
#pragma unroll
                for (int r = 0; r < E; ++r) {
                    const C p = pb[((N - lane - r * R1) & (N - 1)) * W];
                    v[r] = mk<float>(0.5f * (v[r].x + p.x), 0.5f * (v[r].y - p.y));
                }
            }
        }
        C *out = (a.state_out ? a.state_out : a.state) + ofs;
        if (writes) {
#pragma unroll
            for (int r = 0; r < E; ++r) out[(lane + r * R1) * W] = !planes || kx < sp.hx ? v[r] : mk<float>(0, 0);
        }
        if (MODE == R3_FWD || !inverse) return;
        __syncthreads();                                         // the exchange buffer is free again
    } else {
#pragma unroll
        for (int r = 0; r < E; ++r) {
            v[r] = ok && kept_pos(r) ? a.state[ofs + (lane + r * R1) * W] : mk<float>(0, 0);
        }
    }
    // ---- the inverse of the de-aliased, 1 / N_sites-scaled field
#pragma unroll
    for (int r = 0; r < E; ++r) {
        v[r] = kept_pos(r) ? cscale<float>(v[r], sp.inv_nsites) : mk<float>(0, 0);
    }
    dft_reg<E, +1, float>(v);
#pragma unroll
    for (int r = 0; r < E; ++r) xb[(lane * (E + 1) + r) * W] = v[r];
    __syncthreads();
    const C *TWI = TW + (R1 == E ? 0 : N);
    C *__restrict__ out = a.out + ofs;
    const bool stores = writes && (full || tile * W <= fp.kmax[0]);
#pragma unroll
    for (int s = 0; s < S::BPT; ++s) {
        const int i = lane + s * R1;
        C u[R1];
#pragma unroll
        for (int r = 0; r < R1; ++r) {
            u[r] = xb[(i + r * (E + 1)) * W];
            if (r > 0) {
                const C w = TWI[(r - 1) * E + i];
                u[r] = cmul<float>(u[r], mk<float>(w.x, -w.y));
            }
        }
        dft_reg<R1, +1, float>(u);
        if (stores) {
#pragma unroll
            for (int r = 0; r < R1; ++r) out[(i + r * E) * W] = u[r];
        }
    }
}

// The y pass of one tile and PZ z-planes (F = PZ W transforms, PZ >= 4: a half
// warp's accesses are one row of the exchange buffer).
template <int N, int DIR> __global__ void __launch_bounds__(256, 3) k3_mid(const MidArgs<float> a) {
    using S = R3Shape<N>;
    using C = float2;
    constexpr int E = S::E, R1 = S::R1;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    C *TW = reinterpret_cast<C *>(smem_raw);
    C *XCH = TW + S::TWN;
    const SysP<float> &sp = a.sp;
    const int F = a.PZ * W, logF = __ffs(F) - 1;
    const int t = threadIdx.x, f = t & (F - 1), lane = t >> logF;
    const int slot = a.slot0 + blockIdx.z, tile = blockIdx.x;
    r3_twiddles<N>(TW, a.tw, t, blockDim.x);
    const int kmy = a.mode == MID_INV_MASK ? a.fps[slot].kmax[1] : N;
    const uint32_t ostride = (uint32_t)sp.nz * W;               // (a field has fewer than 2^32 values)
    const size_t ofs = (size_t)slot * a.slot_stride + (size_t)tile * N * ostride + (size_t)blockIdx.y * F + f;
    const C *__restrict__ in = a.in + ofs;
    C *__restrict__ out = a.out + ofs;
    pdl_wait();
    pdl_trigger();
    C v[E];
#pragma unroll
    for (int s = 0; s < S::BPT; ++s)
#pragma unroll
        for (int r = 0; r < R1; ++r) {
            const uint32_t p = lane + s * R1 + r * E;
            v[s * R1 + r] = DIR < 0 || abs(signed_k((int)p, N)) <= kmy ? in[p * ostride] : mk<float>(0, 0);
        }
#pragma unroll
    for (int s = 0; s < S::BPT; ++s) {
        dft_reg<R1, DIR, float>(v + s * R1);
#pragma unroll
        for (int r = 0; r < R1; ++r) XCH[((lane + s * R1) * R1 + r) * F + f] = v[s * R1 + r];
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < E; ++r) {
        v[r] = XCH[(lane + r * R1) * F + f];
        if (r > 0) {
            C w = TW[(r - 1) * R1 + lane];
            if (DIR > 0) w.y = -w.y;
            v[r] = cmul<float>(v[r], w);
        }
    }
    dft_reg<E, DIR, float>(v);
#pragma unroll
    for (int r = 0; r < E; ++r) out[(uint32_t)(lane + r * R1) * ostride] = v[r];
    if (a.inc_step && blockIdx.x == 0 && blockIdx.y == 0 && blockIdx.z == 0 && t == 0) *a.d_step += 1;
}

// The x pass: pairs of rows a, b on one complex transform z = a + i b, as in
// k_row (C2R of Z_k = A_k + i B_k, the power, R2C with A_k = (W_k + conj
// W_{N-k}) / 2, B_k = (W_k - conj W_{N-k}) / (2i)).  The R1 threads of a pair
// are neighbours in one warp, so its exchanges need no CTA barrier, and the
// mirrored modes N - k change hands by shuffles: thread `lane` holds modes
// lane + s R1 + r E, whose mirrors are thread R1 - lane's in reverse order
// (thread 0's are its own, one further on).
enum { R3_FUSED = 0, R3_R2C = 1, R3_C2R = 2 };

template <int N> struct R3Row {
    using S = R3Shape<N>;
    // exchange buffer of a pair: the pairs of a half warp fall in different banks
    static constexpr int BUF = (N + S::E + 15) / 16 * 16 + S::R1 % 16;
    // index of mode N - k of thread 0, k at s R1 + r
    static constexpr __host__ __device__ int own(int s, int r) {
        return s == 0 ? (S::R1 - r) % S::R1 : (S::BPT - s) * S::R1 + S::R1 - 1 - r;
    }
};

// A thread's place in the x pass: its transform lane, its pair's exchange
// buffer, and the twiddles.
template <int N> struct R3Line {
    using S = R3Shape<N>;
    using C = float2;
    static constexpr int E = S::E, R1 = S::R1, H = R1 / 2;
    int lane, mirror;
    uint32_t rows, r0;                                           // rows r0 and r0 + 1 of `rows`
    bool ok;
    C *xb;
    const C *TW;

    __device__ __forceinline__ R3Line(int t, int rows_, int r0_, C *xb_, const C *TW_)
        : lane(t % R1), mirror((t & 31 & ~(R1 - 1)) | ((R1 - t % R1) & (R1 - 1))), rows((uint32_t)rows_),
          r0((uint32_t)r0_), ok(r0_ < rows_), xb(xb_), TW(TW_) {}
    // mode lane + s R1 + r E of row r0 (row r0 + 1: W further on); a field has fewer than 2^32 values
    __device__ __forceinline__ uint32_t ofs(int s, int r) const {
        const int k = lane + s * R1 + r * E;
        return ((uint32_t)(k >> 2) * rows + r0) * W + (uint32_t)(k & (W - 1));
    }
    // the two rows of a half spectrum (modes below kxc; dx: times i q_x, 0 at the
    // Nyquist index) -> sites lane + r R1 of both
    __device__ __forceinline__ void to_real(C *v, const C *__restrict__ in, int kxc, bool dx, float gx) const {
        C m[E / 2];                                              // Z_{N-k} for the thread that holds it
#pragma unroll
        for (int s = 0; s < S::BPT; ++s)
#pragma unroll
            for (int r = 0; r < H; ++r) {
                C A = mk<float>(0, 0), B = A;
                const int k = lane + s * R1 + r * E;
                if (ok && k < kxc) {
                    const uint32_t p = ofs(s, r);
                    A = in[p];
                    B = in[p + W];
                    if (dx) {
                        const float q = (float)k * gx;
                        A = mk<float>(-q * A.y, q * A.x);
                        B = mk<float>(-q * B.y, q * B.x);
                    }
                    if (s == 0 && r == 0 && lane == 0) A.y = B.y = 0.0f;
                }
                v[s * R1 + r] = mk<float>(A.x - B.y, A.y + B.x);
                m[s * H + r] = mk<float>(A.x + B.y, B.x - A.y);
            }
#pragma unroll
        for (int s = 0; s < S::BPT; ++s)
#pragma unroll
            for (int r = H; r < R1; ++r) {
                const C x = m[(S::BPT - 1 - s) * H + R1 - 1 - r];
                C z = mk<float>(__shfl_sync(0xffffffffu, x.x, mirror), __shfl_sync(0xffffffffu, x.y, mirror));
                if (s == 0 && r == H) {
                    if (lane == 0) {
                        z = mk<float>(0, 0);
                        if (ok && N / 2 < kxc && !dx) {
                            const uint32_t p = ofs(0, H);
                            z = mk<float>(in[p].x, in[p + W].x);
                        }
                    }
                } else if (lane == 0) {
                    z = m[s == 0 ? R1 - r : (S::BPT - s) * H + R1 - 1 - r];
                }
                v[s * R1 + r] = z;
            }
        __syncwarp();                                            // the buffer is free
#pragma unroll
        for (int s = 0; s < S::BPT; ++s) {
            dft_reg<R1, +1, float>(v + s * R1);
#pragma unroll
            for (int r = 0; r < R1; ++r) xb[(lane + s * R1) * (R1 + 1) + r] = v[s * R1 + r];
        }
        __syncwarp();
#pragma unroll
        for (int r = 0; r < E; ++r) {
            v[r] = xb[lane + r * (R1 + 1)];
            if (r > 0) {
                const C w = TW[(r - 1) * R1 + lane];
                v[r] = cmul<float>(v[r], mk<float>(w.x, -w.y));
            }
        }
        dft_reg<E, +1, float>(v);
    }
    // sites lane + r R1 of both rows -> their half spectra
    __device__ __forceinline__ void to_modes(C *v, C *__restrict__ out) const {
        const C *TWI = TW + (R1 == E ? 0 : N);
        dft_reg<E, -1, float>(v);
        __syncwarp();                                            // the buffer is free
#pragma unroll
        for (int r = 0; r < E; ++r) xb[lane * (E + 1) + r] = v[r];
        __syncwarp();
#pragma unroll
        for (int s = 0; s < S::BPT; ++s) {
            const int i = lane + s * R1;
#pragma unroll
            for (int r = 0; r < R1; ++r) {
                v[s * R1 + r] = xb[i + r * (E + 1)];
                if (r > 0) v[s * R1 + r] = cmul<float>(v[s * R1 + r], TWI[(r - 1) * E + i]);
            }
            dft_reg<R1, -1, float>(v + s * R1);
        }
#pragma unroll
        for (int s = 0; s < S::BPT; ++s)
#pragma unroll
            for (int r = 0; r < H; ++r) {
                const C x = v[s * R1 + r], y = v[E - 1 - (s * R1 + r)];
                C z = mk<float>(__shfl_sync(0xffffffffu, y.x, mirror), __shfl_sync(0xffffffffu, y.y, mirror));
                if (lane == 0) z = v[R3Row<N>::own(s, r)];
                if (ok) {
                    const uint32_t p = ofs(s, r);
                    out[p] = mk<float>(0.5f * (x.x + z.x), 0.5f * (x.y - z.y));
                    out[p + W] = mk<float>(0.5f * (x.y + z.y), -0.5f * (x.x - z.x));
                }
            }
        if (ok && lane < W) {                                    // mode N / 2 and the last tile's padding
            const uint32_t p = ofs(0, H);
            out[p] = mk<float>(lane == 0 ? v[H].x : 0.0f, 0.0f);
            out[p + W] = mk<float>(lane == 0 ? v[H].y : 0.0f, 0.0f);
        }
    }
};

template <int N, int MODE> __global__ void __launch_bounds__(128, R3Shape<N>::CTAS) k3_row(const RowArgs<float> a) {
    using S = R3Shape<N>;
    using C = float2;
    constexpr int E = S::E, R1 = S::R1;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    C *TW = reinterpret_cast<C *>(smem_raw);
    const SysP<float> &sp = a.sp;
    const int t = threadIdx.x, g = t / R1, r0 = 2 * (blockIdx.x * a.G + g);
    const R3Line<N> line(t, sp.rows, r0, TW + S::TWN + g * R3Row<N>::BUF, TW);
    const int slot = a.slot0 + blockIdx.y;
    const size_t sofs = (size_t)slot * a.slot_stride;
    r3_twiddles<N>(TW, a.tw, t, blockDim.x);
    __syncthreads();
    pdl_wait();
    pdl_trigger();
    C v[E];
    if constexpr (MODE != R3_R2C)
        line.to_real(v, a.in + sofs, MODE == R3_FUSED ? a.fps[slot].kx_cols : sp.hx, false, 0.0f);
    if constexpr (MODE == R3_FUSED) {
        const int p = a.fps[slot].power;
        if (p == 3) {
#pragma unroll
            for (int r = 0; r < E; ++r) v[r] = mk<float>(v[r].x * v[r].x * v[r].x, v[r].y * v[r].y * v[r].y);
        } else {
#pragma unroll
            for (int r = 0; r < E; ++r) v[r] = mk<float>(ipow<float>(v[r].x, p), ipow<float>(v[r].y, p));
        }
    } else if (line.ok) {
        const size_t ra = (size_t)slot * a.real_stride + real_row_offset(sp, r0) + line.lane;
        const size_t rb = (size_t)slot * a.real_stride + real_row_offset(sp, r0 + 1) + line.lane;
#pragma unroll
        for (int r = 0; r < E; ++r) {
            if (MODE == R3_C2R) {
                a.real_out[ra + r * R1] = v[r].x;
                a.real_out[rb + r * R1] = v[r].y;
            } else {
                v[r] = mk<float>(a.real_in[ra + r * R1], a.real_in[rb + r * R1]);
            }
        }
    } else if (MODE == R3_R2C) {
#pragma unroll
        for (int r = 0; r < E; ++r) v[r] = mk<float>(0, 0);
    }
    if constexpr (MODE != R3_C2R) {
        line.to_modes(v, a.out + sofs);
        if (a.inc_step && blockIdx.x == 0 && blockIdx.y == 0 && t == 0) *a.d_step += 1;
    }
}

// The x pass of product terms (k_row_terms) on the same lines, 2D rows of up to
// 256 points: every distinct factor's rows to real space (kept in shared memory,
// each thread its own sites), then per target field the sum of its terms and
// back.  No CTA barrier after the twiddles.  us per step, k_row_terms -> here: a
// coupled pair at 256^2 19.2 -> 14.6, at 64^2 16.5 -> 10.3, KPZ at 64^2 16.3 ->
// 12.8, at 256 x 64 17.8 -> 15.6.  Above 256 points a thread would hold 32 sites
// of a chain of transforms and too few warps are left to hide it.
template <int N> __global__ void __launch_bounds__(128, 4) k3_terms(const TermArgs a) {
    using S = R3Shape<N>;
    using C = float2;
    constexpr int E = S::E, R1 = S::R1;
    extern __shared__ __align__(128) unsigned char smem_raw[];
    C *TW = reinterpret_cast<C *>(smem_raw);
    const SysP<float> &sp = a.sp;
    const TermProg &pg = a.prog;
    const int t = threadIdx.x, g = t / R1;
    C *R = TW + S::TWN + a.G * R3Row<N>::BUF + (size_t)g * pg.nfac * N + t % R1;   // [factor][site]
    const R3Line<N> line(t, sp.rows, 2 * (blockIdx.x * a.G + g), TW + S::TWN + g * R3Row<N>::BUF, TW);
    const int slot0 = blockIdx.y * a.nf;
    r3_twiddles<N>(TW, a.tw, t, blockDim.x);
    __syncthreads();
    pdl_wait();
    pdl_trigger();
    C v[E];
#pragma unroll 1
    for (int f = 0; f < pg.nfac; ++f) {
        const TermFactor fc = pg.fac[f];
        const int slot = slot0 + fc.field;
        line.to_real(v, (fc.arr < 0 ? a.in : a.extra + (size_t)fc.arr * a.extra_stride) + (size_t)slot * a.slot_stride,
                     a.fps[slot].kx_cols, fc.dx != 0, sp.gx);
#pragma unroll
        for (int r = 0; r < E; ++r) R[f * N + r * R1] = v[r];
    }
#pragma unroll 1
    for (int f = 0; f < a.nf; ++f) {
        if (pg.nterm[f] == 0) continue;
        const float *coef = a.coef + (size_t)(slot0 + f) * kMaxTerms;
#pragma unroll
        for (int r = 0; r < E; ++r) v[r] = mk<float>(0, 0);
#pragma unroll 1
        for (int i = 0; i < pg.nterm[f]; ++i) {
            const TermP &tm = pg.term[f][i];
            C p[E];
#pragma unroll
            for (int r = 0; r < E; ++r) p[r].x = p[r].y = coef[i];
#pragma unroll 1
            for (int k = 0; k < tm.n; ++k) {
                const C *x = R + tm.fac[k] * N;
#pragma unroll 1
                for (int e = 0; e < tm.power[k]; ++e) {
#pragma unroll
                    for (int r = 0; r < E; ++r) {
                        const C y = x[r * R1];
                        p[r] = mk<float>(p[r].x * y.x, p[r].y * y.y);
                    }
                }
            }
#pragma unroll
            for (int r = 0; r < E; ++r) v[r] = cadd<float>(v[r], p[r]);
        }
        line.to_modes(v, a.out + (size_t)(slot0 + f) * a.slot_stride);
    }
    if (a.inc_step && blockIdx.x == 0 && blockIdx.y == 0 && t == 0) *a.d_step += 1;
}

template <int N> cudaError_t launch_terms3_n(const TermArgs &a, int batch, cudaStream_t st) {
    using S = R3Shape<N>;
    const int threads = a.G * S::R1;
    if (threads % 32 || threads > 128 || a.sp.rows % 2 || a.prog.nfac < 1 || a.prog.nfac > kMaxTermFactors)
        return cudaErrorInvalidConfiguration;
    const size_t smem = sizeof(float2) * (size_t)(S::TWN + a.G * (R3Row<N>::BUF + a.prog.nfac * N));
    cudaError_t e = ensure_smem(k3_terms<N>, smem);
    if (e != cudaSuccess) return e;
    return launch_pdl(k3_terms<N>, dim3((a.sp.rows / 2 + a.G - 1) / a.G, batch), threads, smem, st, a);
}

template <int N> cudaError_t launch_row3_n(const RowArgs<float> &a, int nslots, cudaStream_t st) {
    using S = R3Shape<N>;
    const int threads = a.G * S::R1;
    if (threads % 32 || threads > 128 || a.sp.rows % 2) return cudaErrorInvalidConfiguration;
    const dim3 grid((a.sp.rows / 2 + a.G - 1) / a.G, nslots);
    const size_t smem = sizeof(float2) * (size_t)(S::TWN + a.G * R3Row<N>::BUF);
    if (a.mode == ROW_FUSED) return launch_pdl(k3_row<N, R3_FUSED>, grid, threads, smem, st, a);
    if (a.mode == ROW_R2C) return launch_pdl(k3_row<N, R3_R2C>, grid, threads, smem, st, a);
    if (a.mode == ROW_C2R) return launch_pdl(k3_row<N, R3_C2R>, grid, threads, smem, st, a);
    return cudaErrorInvalidValue;
}

// a.F: threads per CTA (128 in 3D)
template <int N, int DIM> cudaError_t launch_col3_nd(const ColArgs<float> &a, int nslots, cudaStream_t st) {
    using S = R3Shape<N>;
    constexpr int np = DIM == 3 ? 2 : 1;
    if (a.F > 128 || a.F % 32 || a.F % (np * S::CHUNK) || (DIM == 3 && a.F != 128)) return cudaErrorInvalidConfiguration;
    const int chunks = a.F / S::CHUNK, ctiles = chunks / np;
    const dim3 grid((a.n_tiles + ctiles - 1) / ctiles, np == 2 ? a.sp.ny / 2 + 1 : 1, nslots);
    const size_t base = sizeof(float2) * (size_t)(S::TWN + chunks * S::BUF);
    const size_t xi = S::ALIAS ? 0 : sizeof(float2) * (size_t)chunks * N * W;
    if (a.mode == COL_STEP) return launch_pdl(k3_col<N, R3_STEP, DIM>, grid, a.F, base + xi, st, a);
    if (a.mode == COL_FWD) return launch_pdl(k3_col<N, R3_FWD, DIM>, grid, a.F, base, st, a);
    if (a.mode == COL_INV_MASK || a.mode == COL_INV_FULL) return launch_pdl(k3_col<N, R3_INV, DIM>, grid, a.F, base, st, a);
    return cudaErrorInvalidValue;
}
template <int N> cudaError_t launch_col3_n(const ColArgs<float> &a, int nslots, cudaStream_t st) {
    if constexpr (N <= 256)
        if (a.sp.dim == 3) return launch_col3_nd<N, 3>(a, nslots, st);
    return a.sp.dim == 2 ? launch_col3_nd<N, 2>(a, nslots, st) : cudaErrorInvalidValue;
}

template <int N> cudaError_t launch_mid3_n(const MidArgs<float> &a, int nslots, int ntiles, cudaStream_t st) {
    using S = R3Shape<N>;
    const int F = a.PZ * W, threads = F * S::R1;
    if (a.PZ < 4 || (a.PZ & (a.PZ - 1)) || a.sp.nz % a.PZ || threads > 256) return cudaErrorInvalidConfiguration;
    const dim3 grid(ntiles, a.sp.nz / a.PZ, nslots);
    const size_t smem = sizeof(float2) * (size_t)(S::TWN + N * F);
    if (a.mode == MID_FWD) return launch_pdl(k3_mid<N, -1>, grid, threads, smem, st, a);
    return launch_pdl(k3_mid<N, +1>, grid, threads, smem, st, a);
}

}  // namespace pss
