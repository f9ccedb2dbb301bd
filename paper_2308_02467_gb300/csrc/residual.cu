// Float-float refinement residual of the FP32 / TF32 local solves for the common element shapes:
// R = -B^ - A X from the structured operator (eq. hdg_local_mat), with X kept as float-float pairs.
//
// What bounds it: the FP32 pipes.  A float-float multiply-add is 11 or 12 FP32 operations, and GB300
// carries out 39.8e12 FP32 lane operations a second, in scalar or packed f32x2 instructions (measured).  Two
// symmetries of the operator halve the multiply-adds:
//   * the phase matrix is circulant, W[k][l] = wc[(k - l) mod N]: with H = N / 2 and the sums and
//     differences p_l = x_l + x_{l+H}, m_l = x_l - x_{l+H}, the angular sum of all N directions is two
//     H x H products (S_k = sum cp[k-l] p_l, D_k = sum cm[k-l] m_l; y_k = S_k + D_k, y_{k+H} = S_k - D_k),
//     N^2 / 2 multiply-adds instead of N^2;
//   * the LGL derivative is centro-antisymmetric, D[p-q][p-a] = -D[q][a]: a line of n1 nodes splits into
//     its even and odd parts the same way (24 multiply-adds instead of 49 for n1 = 7).
// The sums and differences are exact (TwoSum) or float-float, so the result keeps its ~44 bits.
// A thread therefore owns whole angular sums or whole lines of one column, with the shared operands in
// registers and the coefficients as constant-bank operands: one block per element (several for a small
// batch) takes 8 columns at a time and makes three passes over them in shared memory -- diagonal and
// scattering, x-lines, z-lines with the final residual -- accumulating in float-float.  Eight columns
// (32-byte sectors of a row) leave room for two blocks per SM at p = 6, N = 16, so one block's copies
// and barriers overlap the other's arithmetic; the next chunk's columns arrive by cp.async meanwhile.
// The two halves of each split run side by side in packed f32x2 instructions, half the instructions for the
// same roundings (ff2_fma): with scalar ones the issue slots were 70 % used and the pipe 61 %; now waiting for
// the pipe is the first stall.
// Measured against the general kernel of local.cu (one row and two columns per thread, every sum in full):
// 4096 elements at p = 6, N = 16, adjoint form, 11.2 -> 7.5 ms, packed 6.85 ms; 1247 elements at p = 8, N = 16,
// 9.7 -> 5.6 ms for the first and 12.1 -> 7.2 ms for a later pass; 480 elements at p = 6, N = 16, first pass,
// 0.86 ms.
#include <algorithm>
#include <cstring>

#include "elrt_internal.h"
#include "ff.h"

namespace {

constexpr int kCW = 8;  // columns per pass

// Coefficients of the split sums, as float-float pairs (constant bank)
struct ResTab {
    // d < H: (wc[d] + wc[d + H]) / 2 beside (wc[d] - wc[d + H]) / 2; d + H: the same, the second one negated
    ffc2 W[ELRT_MAX_ANG];
    // [a][q] (wd[q][a] - wd[p-q][a]) / 2, of the difference o_q, beside (wd[q][a] + wd[p-q][a]) / 2, of the sum e_q
    ffc2 UV[5 * 5];
    ff V[5];      // wd[h][a], of the middle node
    ff mid[5];    // wd[q][h]: the middle output takes the differences only
};

// acc = c x and acc += c x, acc left unnormalised (ff.h)
__device__ __forceinline__ ff mul0(ff c, ff x) {
    const float p = __fmul_rn(c.h, x.h);
    float e = fmaf(c.h, x.h, -p);
    e = fmaf(c.h, x.l, e);
    return ff{p, fmaf(c.l, x.h, e)};
}
__device__ __forceinline__ ff mul0(ff c, float x) {
    const float p = __fmul_rn(c.h, x);
    return ff{p, fmaf(c.l, x, fmaf(c.h, x, -p))};
}
__device__ __forceinline__ void mac(ff& acc, ff c, ff x) { ff_fma(acc, c, x); }
__device__ __forceinline__ void mac(ff& acc, ff c, float x) { ff_fma_f(acc, x, c); }
__device__ __forceinline__ ff sum2(float a, float b) {
    ff r;
    two_sum(a, b, r.h, r.l);
    return r;
}
__device__ __forceinline__ ff sum2(ff a, ff b) { return ff_add(a, b); }
__device__ __forceinline__ float neg(float a) { return -a; }
__device__ __forceinline__ ff neg(ff a) { return ff{-a.h, -a.l}; }

// y[k] = sum_l wc[(k - l) mod N] x[l], handed to put(k, y)
template <int N, typename XS, typename Put>
__device__ __forceinline__ void angular(const ResTab& rt, const XS (&x)[N], Put put) {
    constexpr int H = N / 2;
    f2 xh[H], xl[H];  // (sum, difference)
#pragma unroll
    for (int l = 0; l < H; ++l) {
        const ff p = sum2(x[l], x[l + H]), m = sum2(x[l], neg(x[l + H]));
        xh[l] = f2_pack(p.h, m.h);
        xl[l] = f2_pack(p.l, m.l);
    }
#pragma unroll
    for (int k = 0; k < H; ++k) {
        ff2 sd = ff2_mul0(rt.W[k], xh[0], xl[0]);
#pragma unroll
        for (int l = 1; l < H; ++l) ff2_fma(sd, rt.W[k >= l ? k - l : k - l + 2 * H], xh[l], xl[l]);  // cm[d + H] = -cm[d]
        ff s, d;
        ff2_split(sd, s, d);
        put(k, ff_add(s, d));
        put(k + H, ff_add(s, neg(d)));
    }
}

// y[a] = sum_q wd[q][a] x[q] along one line, handed to put(a, y)
template <int N1, typename XS, typename Put>
__device__ __forceinline__ void line(const ResTab& rt, const XS (&x)[N1], Put put) {
    constexpr int h = N1 / 2;
    f2 xh[h], xl[h];  // (difference, sum)
    ff o[h];
#pragma unroll
    for (int q = 0; q < h; ++q) {
        const ff e = sum2(x[q], x[N1 - 1 - q]);
        o[q] = sum2(x[q], neg(x[N1 - 1 - q]));
        xh[q] = f2_pack(o[q].h, e.h);
        xl[q] = f2_pack(o[q].l, e.l);
    }
#pragma unroll
    for (int a = 0; a < h; ++a) {
        ff2 uv = ff2_mul0(rt.UV[a * 5], xh[0], xl[0]);
#pragma unroll
        for (int q = 1; q < h; ++q) ff2_fma(uv, rt.UV[a * 5 + q], xh[q], xl[q]);
        ff u, v;
        ff2_split(uv, u, v);
        mac(v, rt.V[a], x[h]);
        put(a, ff_add(u, v));
        put(N1 - 1 - a, ff_add(u, neg(v)));
    }
    ff c = mul0(rt.mid[0], o[0]);
#pragma unroll
    for (int q = 1; q < h; ++q) mac(c, rt.mid[q], o[q]);
    put(h, ff_norm(c.h, c.l));
}

__device__ __forceinline__ void cp16(void* smem, const void* gmem) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(smem)), "l"(gmem)
                 : "memory");
}

template <int N1, int N, typename XS>
struct ResCfg {
    static constexpr int NM = N1 * N1, NU = NM * N;
    static constexpr bool F = sizeof(XS) == 4;
    // X chunk (and, in the first pass, the next one), accumulators, per-element coefficients
    static constexpr size_t SMEM = (size_t)NU * kCW * (sizeof(XS) + (F ? 4 : 0) + sizeof(ff)) +
                                   ((size_t)NU + NM + 2 * N * N1) * sizeof(ff);
    static constexpr int BLOCKS = SMEM <= 112 * 1024 ? 2 : 1;  // resident blocks per SM
    static constexpr int T = BLOCKS == 2 ? 256 : 512;          // 16 warps per SM either way
    static_assert(SMEM <= 226 * 1024, "residual shared memory");
};

// mode 0: X = D (XS float);  mode 1: X += D (XS ff).  R over D, maxres[e] = max |R|.
// ADJ (XS float, for the adjoint correction of adjoint.cu): the columns of B^ carry the power-of-two scales of
// the assembly (unit_scale of their entry), X = D stays where it is, R goes to Rall
// [E][NU][nin], Xall takes the sums of X over the angular cells [E][NM][nin] instead of X, and no maximum is
// formed.
template <int N1, int N, typename XS, bool ADJ>
__global__ void __launch_bounds__(ResCfg<N1, N, XS>::T, ResCfg<N1, N, XS>::BLOCKS)
    k_residual_eo(const __grid_constant__ Tab t, const __grid_constant__ ResTab rt, double h,
                  const double* __restrict__ h_elem, const double* __restrict__ kappa, const double* __restrict__ omega,
                  float* __restrict__ Mall, int64_t ld, int64_t estride, ff* __restrict__ Xall,
                  double* __restrict__ maxres, float* __restrict__ Rall) {
    using Cfg = ResCfg<N1, N, XS>;
    constexpr int NM = Cfg::NM, NU = Cfg::NU, T = Cfg::T, P = N1 - 1, G = T / kCW;
    constexpr bool F = Cfg::F;
    extern __shared__ __align__(16) unsigned char smem_raw[];
    XS* Xs = reinterpret_cast<XS*>(smem_raw);                 // [NU][kCW]; in the first pass two of them
    ff* Acc = reinterpret_cast<ff*>(Xs + (size_t)(F ? 2 : 1) * NU * kCW);  // [NU][kCW]
    ff* dcoef = Acc + (size_t)NU * kCW;                       // [NU] B^k_ii + w_i kappa_hat_i
    ff* scoef = dcoef + NU;                                   // [NM] -w_i omega kappa_hat_i
    ff* sxw = scoef + NM;                                     // [N][N1] -sx_k w_b
    ff* szw = sxw + N * N1;                                   // [N][N1] -sz_k w_a
    __shared__ float red[T / 32];
    const int nin = t.nin, tid = threadIdx.x;
    const int64_t e = blockIdx.x;
    float* M = Mall + e * estride + NU;  // the right-hand-side columns
    ff* X = Xall + e * (int64_t)(ADJ ? NM : NU) * nin;
    float* Rp = ADJ ? Rall + e * (int64_t)NU * nin : M;
    const int64_t rld = ADJ ? nin : ld;
    // this block's columns: neighbouring chunks, whose rows share cache lines
    const int per = (nin / kCW + gridDim.y - 1) / gridDim.y * kCW;
    const int cs0 = min(nin, (int)blockIdx.y * per), cs1 = min(nin, cs0 + per);
    auto prefetch = [&](int cs, XS* dst) {  // first pass: the chunk's columns of D (two 16-byte halves a row)
        if constexpr (F) {
            for (int q = tid; q < 2 * NU; q += T)
                cp16(dst + (q >> 1) * kCW + (q & 1) * 4, M + (int64_t)(q >> 1) * ld + cs + (q & 1) * 4);
            asm volatile("cp.async.commit_group;" ::: "memory");
        }
    };
    if (cs0 < cs1) prefetch(cs0, Xs);
    const double he = h_elem ? h_elem[e] : h;
    const double om = omega[e];
    for (int q = tid; q < NM; q += T)
        scoef[q] = ff_from_double(-(t.w[q % N1] * t.w[q / N1] * om * kappa[e * NM + q] * 0.5 * he));
    for (int q = tid; q < N * N1; q += T) {
        const int k = q / N1, b = q - k * N1;
        sxw[q] = ff_from_double(-t.sx[k] * t.w[b]);
        szw[q] = ff_from_double(-t.sz[k] * t.w[b]);
    }
    for (int r = tid; r < NU; r += T) {
        const int k = r / NM, i = r - k * NM;
        const int a = i % N1, b = i / N1;
        double bd = 0.0;
        if (b == 0 && t.sdn[0][k] > 0) bd += t.w[a] * t.sdn[0][k];
        if (a == P && t.sdn[1][k] > 0) bd += t.w[b] * t.sdn[1][k];
        if (b == P && t.sdn[2][k] > 0) bd += t.w[a] * t.sdn[2][k];
        if (a == 0 && t.sdn[3][k] > 0) bd += t.w[b] * t.sdn[3][k];
        dcoef[r] = ff_from_double(bd + t.w[a] * t.w[b] * kappa[e * NM + i] * 0.5 * he);
    }
    const int col = tid & (kCW - 1), g = tid / kCW;
    float rmax = 0.f;
    int buf = 0;
    for (int cs = cs0; cs < cs1; cs += kCW, buf ^= 1) {
        const XS* xs = Xs;
        if constexpr (F) {
            asm volatile("cp.async.wait_all;" ::: "memory");
            __syncthreads();  // the chunk has landed; the last pass over the other buffer is done
            xs = Xs + (size_t)buf * NU * kCW;
            if (cs + kCW < cs1) prefetch(cs + kCW, Xs + (size_t)(buf ^ 1) * NU * kCW);
            if constexpr (!ADJ)
                for (int r = g; r < NU; r += G) X[(int64_t)r * nin + cs + col] = ff{xs[r * kCW + col], 0.f};
        } else {
            __syncthreads();
            constexpr int SB = 8;  // independent loads in flight
            for (int rb = g; rb < NU; rb += SB * G) {
                float d[SB];
                ff xo[SB];
#pragma unroll
                for (int u = 0; u < SB; ++u) {
                    const int r = rb + u * G;
                    if (r < NU) {
                        d[u] = M[(int64_t)r * ld + cs + col];
                        xo[u] = X[(int64_t)r * nin + cs + col];
                    }
                }
#pragma unroll
                for (int u = 0; u < SB; ++u) {
                    const int r = rb + u * G;
                    if (r < NU) {
                        const ff v = ff_add(xo[u], ff{d[u], 0.f});
                        X[(int64_t)r * nin + cs + col] = v;
                        Xs[r * kCW + col] = v;
                    }
                }
            }
            __syncthreads();
        }
        // (B + M) X - S X: one node's N directions per unit
        for (int i = g; i < NM; i += G) {
            XS x[N];
#pragma unroll
            for (int l = 0; l < N; ++l) x[l] = xs[(l * NM + i) * kCW + col];
            if constexpr (ADJ) {
                ff m = sum2(x[0], x[1]);
#pragma unroll
                for (int l = 2; l < N; ++l) m = ff_add(m, ff{x[l], 0.f});
                X[(int64_t)i * nin + cs + col] = m;
            }
            const ff sc = scoef[i];
            angular<N>(rt, x, [&](int k, ff y) {
                ff acc = mul0(dcoef[k * NM + i], x[k]);
                mac(acc, sc, y);
                Acc[(k * NM + i) * kCW + col] = acc;
            });
        }
        __syncthreads();
        // - C X along the x-lines
        for (int q = g; q < N * N1; q += G) {
            const int k = q / N1, b = q - k * N1, r0 = k * NM + N1 * b;
            XS x[N1];
#pragma unroll
            for (int a = 0; a < N1; ++a) x[a] = xs[(r0 + a) * kCW + col];
            const ff c = sxw[q];
            line<N1>(rt, x, [&](int a, ff y) {
                ff acc = Acc[(r0 + a) * kCW + col];
                mac(acc, c, y);
                Acc[(r0 + a) * kCW + col] = acc;
            });
        }
        __syncthreads();
        // - C X along the z-lines, and the residual; the one nonzero of this column of B^ is (tr, tv)
        const int c = cs + col, Fc = c / t.nface, rem = c - Fc * t.nface, m = rem / t.half;
        const int kin = t.inc[Fc][rem - m * t.half];
        const int tr = kin * NM + face_node(Fc, m, P);
        ff tv = ff_from_double(-t.w[m] * t.sdn[Fc][kin]);
        if constexpr (ADJ) {
            // the scale the assembly used: the power of two is that of the entry in FP32 arithmetic
            const float us = unit_scale((float)-t.w[m] * (float)t.sdn[Fc][kin]);
            tv = ff{tv.h * us, tv.l * us};
        }
        for (int q = g; q < N * N1; q += G) {
            const int k = q / N1, a = q - k * N1, r0 = k * NM + a;
            XS x[N1];
#pragma unroll
            for (int b = 0; b < N1; ++b) x[b] = xs[(r0 + N1 * b) * kCW + col];
            const ff cz = szw[q];
            line<N1>(rt, x, [&](int b, ff y) {
                const int r = r0 + N1 * b;
                ff acc = Acc[r * kCW + col];
                mac(acc, cz, y);
                acc = ff_norm(acc.h, acc.l);
                const ff res = r == tr ? ff_add(tv, neg(acc)) : neg(acc);
                const float rf = __fadd_rn(res.h, res.l);
                if constexpr (!ADJ) rmax = fmaxf(rmax, fabsf(rf));
                Rp[(int64_t)r * rld + c] = rf;
            });
        }
    }
    if constexpr (ADJ) return;
    for (int off = 16; off > 0; off >>= 1) rmax = fmaxf(rmax, __shfl_down_sync(0xffffffffu, rmax, off));
    if ((tid & 31) == 0) red[tid >> 5] = rmax;
    __syncthreads();
    if (tid == 0) {
        float mx = 0.f;
        for (int w = 0; w < T / 32; ++w) mx = fmaxf(mx, red[w]);
        if (gridDim.y == 1) maxres[e] = (double)mx;
        else  // several blocks per element: the maximum of non-negative doubles by their bit patterns (zeroed first)
            atomicMax(reinterpret_cast<unsigned long long*>(maxres + e), (unsigned long long)__double_as_longlong((double)mx));
    }
}

ResTab make_tab(const Tab& t) {
    ResTab r{};
    const int H = t.N / 2, n1 = t.n1, h = n1 / 2;
    auto pair = [](double a, double b) {
        const ff x = ff_from_double_host(a), y = ff_from_double_host(b);
        auto two = [](float lo, float hi) {
            const float v[2] = {lo, hi};
            f2 r;
            memcpy(&r, v, sizeof(r));
            return r;
        };
        return ffc2{two(x.h, y.h), two(-x.h, -y.h), two(-x.l, -y.l)};
    };
    for (int d = 0; d < H; ++d) {
        const double cp = 0.5 * (t.wc[d] + t.wc[d + H]), cm = 0.5 * (t.wc[d] - t.wc[d + H]);
        r.W[d] = pair(cp, cm);
        r.W[d + H] = pair(cp, -cm);
    }
    auto wd = [&](int q, int a) { return t.w[q] * t.D[q * n1 + a]; };
    for (int a = 0; a < h; ++a) {
        for (int q = 0; q < h; ++q)
            r.UV[a * 5 + q] = pair(0.5 * (wd(q, a) - wd(n1 - 1 - q, a)), 0.5 * (wd(q, a) + wd(n1 - 1 - q, a)));
        r.V[a] = ff_from_double_host(wd(h, a));
        r.mid[a] = ff_from_double_host(wd(a, h));
    }
    return r;
}

struct Args {
    elrt_ctx* ctx;
    double h;
    const double *h_elem, *kappa, *omega;
    float* M;
    int64_t ld, estride;
    ff* X;
    double* maxres;
    float* R;
    int64_t n;
};

template <int N1, int N, typename XS, bool ADJ = false>
elrt_status launch(const Args& a) {
    using Cfg = ResCfg<N1, N, XS>;
    const Tab& t = a.ctx->tab;
    cudaError_t e = cudaFuncSetAttribute(k_residual_eo<N1, N, XS, ADJ>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)Cfg::SMEM);
    if (e != cudaSuccess) return cuda_check(a.ctx, e, "smem attribute");
    // gy blocks share an element's column chunks: as many as make (waves of blocks) x (chunks a block takes,
    // and half a one for its coefficients and its first load) least.  A small batch fills the GPU that way, and a
    // larger one loses less to its last wave: against one block an element, 480 elements (p = 6, N = 16; gy = 5)
    // 1.11 -> 0.86 ms, 1247 (p = 8; gy = 4) 6.18 -> 5.57 ms.  The blocks take neighbouring chunks: taken in turn,
    // 0.94 and 5.87 ms, and the pass that reads X too 8.4 instead of 7.2 (its cache lines came in for each block).
    const int64_t slots = (int64_t)Cfg::BLOCKS * a.ctx->sms;
    const int chunks = t.nin / kCW;
    int gy = 1;
    int64_t least = INT64_MAX;
    for (int y = 1; y <= chunks; ++y) {
        const int64_t cost = ((a.n * y + slots - 1) / slots) * (2 * ((chunks + y - 1) / y) + 1);
        if (cost < least) least = cost, gy = y;
    }
    if (gy > 1 && !ADJ) {
        e = cudaMemsetAsync(a.maxres, 0, (size_t)a.n * sizeof(double), a.ctx->stream);
        if (e != cudaSuccess) return cuda_check(a.ctx, e, "residual maxima");
    }
    k_residual_eo<N1, N, XS, ADJ><<<dim3((unsigned)a.n, (unsigned)gy), Cfg::T, Cfg::SMEM, a.ctx->stream>>>(
        t, make_tab(t), a.h, a.h_elem, a.kappa, a.omega, a.M, a.ld, a.estride, a.X, a.maxres, a.R);
    return cuda_check(a.ctx, cudaGetLastError(), "residual launch");
}

template <int N1, int N>
elrt_status launch_mode(const Args& a, int mode) {
    if (mode == 3) return launch<N1, N, float, true>(a);
    return mode == 0 ? launch<N1, N, float>(a) : launch<N1, N, ff>(a);
}

}  // namespace

// Shapes with a kernel here: p in {2, 4, 6, 8} with 8, 12 or 16 angular cells, and p = 6 with 28, those of the
// workloads.  Each is three compiled instances with its sums unrolled, which is what bounds the list; the split
// itself needs an odd number of nodes per line and an even number of cells.  Others take the general kernel of
// local.cu (and builds of theirs the re-solve).
bool residual_eo_fits(const Tab& t) {
    const bool n = t.N == 8 || t.N == 12 || t.N == 16;
    return (n && (t.n1 == 3 || t.n1 == 5 || t.n1 == 7 || t.n1 == 9)) || (t.n1 == 7 && t.N == 28);
}

elrt_status residual_eo(elrt_ctx* ctx, double h, const double* h_elem, const double* kappa, const double* omega, float* M,
                        int64_t ld, int64_t estride, void* X, int mode, double* maxres, int64_t n, float* R) {
    const Args a{ctx, h, h_elem, kappa, omega, M, ld, estride, (ff*)X, maxres, R, n};
    switch (ctx->tab.n1 * 100 + ctx->tab.N) {
        case 308: return launch_mode<3, 8>(a, mode);
        case 312: return launch_mode<3, 12>(a, mode);
        case 316: return launch_mode<3, 16>(a, mode);
        case 508: return launch_mode<5, 8>(a, mode);
        case 512: return launch_mode<5, 12>(a, mode);
        case 516: return launch_mode<5, 16>(a, mode);
        case 708: return launch_mode<7, 8>(a, mode);
        case 712: return launch_mode<7, 12>(a, mode);
        case 716: return launch_mode<7, 16>(a, mode);
        case 728: return launch_mode<7, 28>(a, mode);
        case 908: return launch_mode<9, 8>(a, mode);
        case 912: return launch_mode<9, 12>(a, mode);
        case 916: return launch_mode<9, 16>(a, mode);
    }
    return ctx_fail(ctx, ELRT_EINVAL, "residual: unsupported element shape");
}
