// The last refinement step of a TF32_IR build whose caller wants the FP32 operators alone (no statistics, no
// status words, no A_i2u): the correction R A^{-1} r of the restricted operators by an adjoint product instead of a
// re-solve of the whole system.  (FP32_IR, whose products stay on the CUDA cores, keeps the re-solve.)
//
// With the residual r = -B^ - A X (float-float, residual.cu) the refined operators are in2out = R^o X +
// R^o A^{-1} r and in2sol = R^m X + R^m A^{-1} r.  The discrete transport operator is reciprocal: with P the
// reversal of every direction (angular cell k <-> k + N/2), A^T = P A P (the collocated derivative satisfies
// summation by parts, upwind faces swap roles under the reversal, and the phase matrix is symmetric).  So
//   R^o A^{-1} = (P A^{-1} P R^oT)^T,  and P R^oT is the -B^ matrix up to its one factor per column: an outflow
//   value's reversal is the inflow column of the same face node -- its solution is already among the columns
//   of X;
//   R^m A^{-1} = (1/N) (P A^{-1} E)^T, E the (p+1)^2 isotropic unit sources, E[(k, i)][i'] = 1 for i = i': the
//   factorisation solves them as extra columns Z.
// Both are the product G = (P [X | Z])^T r, of 2 nu (n_in + nm) n_in flops per element against 2 nu^2 n_in of
// the re-solve and its passes over the matrix.  [X | Z] has the factorisation's accuracy, which multiplies a
// residual of that size, so the refined operators are as accurate as with a re-solve -- provided the columns
// of X are accurate relative to their own size: the assembly scales each -B^ column by a power of two so that
// its entry lies in [0.5, 1), and the epilogue takes the scales out again (without, the 3xFP16 factorisation
// left a thick element's grazing columns thirteen times less accurate than the re-solve).  Before the rounding
// to FP32 it leaves more than a re-solve does: on 256 elements of the slab (p = 6, N = 16) at most 2.7e-11 in in2out
// and 6.8e-12 in in2sol where the re-solve leaves 6.4e-12 and 4.2e-13, since its second factor has the 3xFP16
// factorisation's backward sweep (with 3xTF32 factors 2.4e-12 and 3.3e-13 against 1.4e-12 and 6.0e-14).  The rounded
// operators' largest and mean-square errors are the same to three digits, 5.9e-8 and 1.1e-9; entries below
// ~1e-3 carry the difference.  FP64 operators keep the re-solve.
//
// k_adjoint: one CTA per (element, tile of up to 128 of the n_in columns of r): D[j][c] = sum_rows r[row][j]
// XZ[reversed row][c] in 3xTF32 on the tensor cores (FP32 values are their own high part; the full FP32 range,
// so no scaling), j on the 128 lanes, c on up to 512 columns of tensor memory.  Both operands lie row-major
// with the summation index outermost, so fifteen warps load them with 16-byte loads (four rows of four
// columns a lane), transpose in registers and write K-major, 128-byte-swizzled tiles of 32 rows of the sum,
// eight lanes on one row's eight chunks (no bank conflicts); one thread of a sixteenth warp issues the MMAs.
// Bound by the latency of its loads (about 2.4 MB per element in two column tiles, the second tile's mostly
// from L2; DRAM 25 % and the tensor pipe 28 % busy): 16 warps and two stages of 106 KB are what one SM holds.
// The epilogue reads X at the outflow rows, adds the correction and rounds once.  Measured, builds with one
// refinement step: 4096 elements at p = 6, N = 16, 61.9 -> 51.6 ms (the re-solve and the float-float restriction
// gone, k_adjoint 4.4 ms, the 49 columns 2 ms), 50.8 ms with its loads as below; nine elements 1.92 -> 1.28 ms
// (141 -> 90 launches).
#include <algorithm>

#include "elrt_internal.h"
#include "ff.h"
#include "tc_gemm.cuh"

namespace {

constexpr int kAdjWarps = 15;                      // operand warps
constexpr int kAdjThreads = 32 * (kAdjWarps + 1);  // and the MMA warp; all sixteen run the epilogue
constexpr int kAdjK = 32;                          // rows of the sum per stage: 128 bytes of FP32
// tables of the columns (xrow, orow, scale, us below); with the barriers they are the kernel's static shared
// memory, which the stages' alignment rounds up to 1 KB (ptxas: 10,240 bytes).  The rest of the 227 KB a block
// can have holds the stages
constexpr int kAdjCols = 4 * ELRT_MAX_N1 * ELRT_MAX_ANG / 2;
constexpr int kAdjStatic = (kAdjCols * (int)(sizeof(int) + sizeof(short) + 2 * sizeof(float)) + 64 + 1023) / 1024 * 1024;
constexpr int kAdjSmem = 227 * 1024 - kAdjStatic;
// dynamic shared memory of a launch with that many stages and nc columns (1024: the stages' alignment)
constexpr int adj_smem(int stages, int nc) { return stages * 2 * 128 * (128 + nc) + 1024; }
static_assert(adj_smem(1, 512) <= kAdjSmem, "one stage of the widest product fits");

struct AdjArgs {
    const float* M;        // [E][nu][ld], solution columns from nu: X, then Z
    int64_t ld, estride;
    const float* R;        // [E][nu][nin] residual
    const ff* sum;         // [E][nm][nin] sum over the angular cells of X
    ff inv_n;              // 1 / N
    int jtiles, jw;        // column tiles of r per element, and their width (a multiple of 16)
    int nc;                // n_in + nm rounded up to 16
    int stages;
    int* err;
};

__host__ __device__ constexpr uint32_t adj_idesc(int n) {  // kind::tf32, M = 128
    return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(n >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
}

__device__ __forceinline__ void mma_tf32_ss(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                            uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(
            d_tmem),
        "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate));
}

// column of operand row w within blocks of 16
__host__ __device__ constexpr int unperm16(int w) { return (w & ~15) | (4 * (w & 3) + ((w >> 2) & 3)); }

__global__ void __launch_bounds__(kAdjThreads, 1)
    k_adjoint(const __grid_constant__ Tab t, const __grid_constant__ AdjArgs g, float* __restrict__ in2out,
              float* __restrict__ in2sol) {
    extern __shared__ __align__(1024) unsigned char raw[];
    unsigned char* base = (unsigned char*)(((uintptr_t)raw + 1023) & ~(uintptr_t)1023);
    const int NC = g.nc, NS = g.stages, nin = t.nin, nu = t.nu, nm = t.nm;
    // a stage: r tile high and low (128 rows of 128 bytes each), XZ tile high and low (NC rows each)
    const int a_bytes = 128 * 128, b_bytes = NC * 128, stage = 2 * (a_bytes + b_bytes);
    __shared__ uint64_t full[2], empty[2], acc_full;
    __shared__ uint32_t tmem_slot;
    __shared__ int abort_s;
    __shared__ int xrow[kAdjCols];    // row of X at the outflow value of column c
    __shared__ short orow[kAdjCols];  // its row of in2out
    __shared__ float scale[kAdjCols]; // 1 / the column's (scaled) entry of -B^
    __shared__ float us[kAdjCols];    // 1 / the column's power-of-two scale
    volatile int* abort = &abort_s;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int64_t e = blockIdx.x / g.jtiles;
    const int j0 = (int)(blockIdx.x - e * g.jtiles) * g.jw;
    const int nch = (nu + kAdjK - 1) / kAdjK;
    uint32_t tcols = 32;
    while ((int)tcols < NC) tcols <<= 1;
    if (threadIdx.x == 0) {
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(&full[i], kAdjWarps);
            tc::mbar_init(&empty[i], 1);
        }
        tc::mbar_init(&acc_full, 1);
        abort_s = 0;
        tc::fence_barrier_init();
    }
    if (warp == kAdjWarps) {
        tc::tmem_alloc(&tmem_slot, tcols);
        tc::tmem_relinquish();
    }
    for (int c = threadIdx.x; c < nin; c += kAdjThreads) {
        const int F = c / t.nface, rem = c - F * t.nface, m = rem / t.half, kin = t.inc[F][rem - m * t.half];
        const int kout = kin < t.half ? kin + t.half : kin - t.half;
        int kk = 0;
        while (kk < t.half - 1 && t.outc[F][kk] != kout) ++kk;
        xrow[c] = kout * nm + face_node(F, m, t.p);
        orow[c] = (short)(F * t.nface + m * t.half + kk);
        const float u = unit_scale((float)-t.w[m] * (float)t.sdn[F][kin]);
        scale[c] = (float)(1.0 / (-t.w[m] * t.sdn[F][kin] * u));
        us[c] = 1.f / u;
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    const uint32_t tmem = tmem_slot;
    const float* Me = g.M + e * g.estride + nu;
    const float* Re = g.R + e * (int64_t)nu * nin;
    bool ok = true;
    if (warp < kAdjWarps) {
        // operand tasks of a chunk: 16 columns each, the jw columns of r first, then the nc of XZ; lane: rows
        // 4 kc .. 4 kc + 3 of the chunk, columns 4 c4 .. 4 c4 + 3 of the task.  Four neighbouring lanes read 64
        // bytes of a row (eight rows to eight neighbouring lanes cost four times the L1 wavefronts: k_adjoint
        // 4.8 against 4.4 ms for 4096 elements); with kc and kc + 4 in a quarter warp and column 4 c4 + q in
        // operand row 4 q + c4 of its block of 16 (unperm16), the stores of a quarter touch every bank once.
        const int kc = (lane >> 3) + (lane & 4), c4 = lane & 3;
        const int ja = g.jw / 16, ntask = ja + NC / 16, half = nu / 2, ld = (int)g.ld;
        int swz[4];  // byte offset of this lane's chunk for its column q, within the task's 16 rows
#pragma unroll
        for (int q = 0; q < 4; ++q) swz[q] = (4 * q + c4) * 128 + ((kc ^ ((4 * q + c4) & 7)) << 4);
        auto load = [&](int task, int k0, float4 (&v)[4]) {
            const bool isr = task < ja;
            const int col = 16 * (isr ? task : task - ja) + 4 * c4;
            const bool in = isr ? j0 + col < nin : col < nin + nm;
            const float* p = isr ? Re + j0 + col : Me + col;
            const int rld = isr ? nin : ld;
            const int k = k0 + 4 * kc;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                v[q] = make_float4(0.f, 0.f, 0.f, 0.f);
                // XZ: the reversed direction's row
                const int row = isr ? k + q : (k + q < half ? k + q + half : k + q - half);
                if (in && k + q < nu) v[q] = __ldg(reinterpret_cast<const float4*>(p + row * rld));
            }
        };
        auto store = [&](unsigned char* st, int task, const float4 (&v)[4]) {
            const bool isr = task < ja;
            unsigned char* hi = st + (isr ? task * 2048 : 2 * a_bytes + (task - ja) * 2048);  // 16 rows a task
            const int lo = isr ? a_bytes : b_bytes;
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                float4 x;
                if (q == 0) x = make_float4(v[0].x, v[1].x, v[2].x, v[3].x);
                if (q == 1) x = make_float4(v[0].y, v[1].y, v[2].y, v[3].y);
                if (q == 2) x = make_float4(v[0].z, v[1].z, v[2].z, v[3].z);
                if (q == 3) x = make_float4(v[0].w, v[1].w, v[2].w, v[3].w);
                auto low = [](float f) { return f - __uint_as_float(__float_as_uint(f) & 0xFFFFE000u); };
                *reinterpret_cast<float4*>(hi + swz[q]) = x;
                *reinterpret_cast<float4*>(hi + swz[q] + lo) = make_float4(low(x.x), low(x.y), low(x.z), low(x.w));
            }
        };
        // the next chunk's first two tasks are loaded before this chunk's are stored, so their latency passes
        // behind the wait for the stage, the stores and the MMAs (5.0 -> 4.8 ms)
        auto load2 = [&](int ch, float4 (&v)[2][4]) {
#pragma unroll
            for (int u = 0; u < 2; ++u)
                if (ch < nch && warp + u * kAdjWarps < ntask) load(warp + u * kAdjWarps, ch * kAdjK, v[u]);
        };
        auto chunk = [&](int ch, const float4 (&v)[2][4], float4 (&next)[2][4]) {
            const int s = ch % NS;
            unsigned char* st = base + s * stage;
            load2(ch + 1, next);
            // the stage is free (a warp without a task waits too: one arrival per phase)
            ok = __all_sync(0xffffffffu, tc::mbar_wait(&empty[s], ((ch / NS) & 1) ^ 1, abort) && !*abort);
            if (!ok) return;
#pragma unroll
            for (int u = 0; u < 2; ++u)
                if (warp + u * kAdjWarps < ntask) store(st, warp + u * kAdjWarps, v[u]);
            for (int task = warp + 2 * kAdjWarps; task < ntask; task += kAdjWarps) {  // (wide elements)
                float4 w[4];
                load(task, ch * kAdjK, w);
                store(st, task, w);
            }
            tc::fence_proxy_async();  // written through the generic proxy, read by the MMAs (async proxy)
            __syncwarp();
            if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(tc::smem_u32(&full[s])) : "memory");
        };
        float4 va[2][4], vb[2][4];
        load2(0, va);
        for (int ch = 0; ch < nch && ok; ch += 2) {
            chunk(ch, va, vb);
            if (ok && ch + 1 < nch) chunk(ch + 1, vb, va);
        }
    } else {
        if (lane == 0) {
            const int n0 = min(NC, 256), n1 = NC - n0;
            const uint32_t id0 = adj_idesc(n0), id1 = adj_idesc(n1);
            uint32_t acc = 0;
            int done = 0;
            for (int ch = 0; ch < nch; ++ch) {
                const int s = ch % NS;
                if (!tc::mbar_wait(&full[s], (ch / NS) & 1, abort)) {
                    ok = false;
                    break;
                }
                tc::tc_fence_after();
                const uint32_t st = tc::smem_u32(base + s * stage);
                const uint64_t ah = tc::sw128_desc(st), al = tc::sw128_desc(st + a_bytes);
                const uint64_t bh = tc::sw128_desc(st + 2 * a_bytes), bl = tc::sw128_desc(st + 2 * a_bytes + b_bytes);
                const uint64_t b1 = 256 * 128 / 16;  // the columns from 256 on
#pragma unroll
                for (int k = 0; k < kAdjK / 8; ++k) {  // K = 8 per instruction: 32 bytes
                    mma_tf32_ss(tmem, ah + 2 * k, bh + 2 * k, id0, acc);
                    if (n1) mma_tf32_ss(tmem + 256, ah + 2 * k, bh + b1 + 2 * k, id1, acc);
                    acc = 1;
                    mma_tf32_ss(tmem, al + 2 * k, bh + 2 * k, id0, 1);
                    if (n1) mma_tf32_ss(tmem + 256, al + 2 * k, bh + b1 + 2 * k, id1, 1);
                    mma_tf32_ss(tmem, ah + 2 * k, bl + 2 * k, id0, 1);
                    if (n1) mma_tf32_ss(tmem + 256, ah + 2 * k, bl + b1 + 2 * k, id1, 1);
                }
                tc::mma_commit(&empty[s]);
                ++done;
            }
            if (!ok) {
                atomicOr(g.err, 8192);
                *abort = 1;
            }
            tc::mma_commit(&acc_full);
            // every MMA has completed before the tensor memory and the barriers go (bounded)
            const long long t0 = clock64();
            while (!tc::mbar_try_wait(&acc_full, 0) && clock64() - t0 < tc::kWaitCycles) {
            }
            for (int ch = max(0, done - NS); ch < done; ++ch)
                while (!tc::mbar_try_wait(&empty[ch % NS], (ch / NS) & 1) && clock64() - t0 < tc::kWaitCycles) {
                }
        }
        __syncwarp();
    }
    // epilogue: lane j of the accumulator, 16 columns at a time, four warps per lane quarter
    {
        const int quad = warp & 3, jl = 32 * quad + unperm16(lane), j = j0 + jl;
        const bool jin = jl < g.jw && j < nin;
        ok = __all_sync(0xffffffffu, ok && tc::mbar_wait(&acc_full, 0, abort) && !*abort);
        if (ok) {
            tc::tc_fence_after();
            const float uj = jin ? us[j] : 1.f;
            const ff* se = g.sum + e * (int64_t)nm * nin;
            float* oo = in2out + e * (int64_t)nin * nin;
            float* om = in2sol + e * (int64_t)nm * nin;
            for (int b = warp >> 2; b < NC / 16; b += 4) {
                float x[16], d[16];
                const int cb = 16 * b;
#pragma unroll
                for (int q = 0; q < 16; ++q) {
                    const int c = cb + unperm16(q);
                    x[q] = (jin && c < nin) ? Me[(int64_t)xrow[c] * g.ld + j] : 0.f;
                }
                tc::tmem_ld16(tmem + ((uint32_t)(32 * quad) << 16) + (uint32_t)cb, d);
                if (jin) {
#pragma unroll
                    for (int q = 0; q < 16; ++q) {
                        const int c = cb + unperm16(q);
                        if (c < nin) {
                            oo[(int64_t)orow[c] * nin + j] = __fadd_rn(x[q] * uj, d[q] * (scale[c] * uj));
                        } else if (c < nin + nm) {
                            const int i = c - nin;
                            const ff v = ff_mul(ff_add(se[(int64_t)i * nin + j], ff{d[q], 0.f}), g.inv_n);
                            om[(int64_t)i * nin + j] = __fadd_rn(v.h * uj, v.l * uj);
                        }
                    }
                }
            }
        }
        if (!ok && lane == 0) {
            atomicOr(g.err, 4096);
            *abort = 1;
        }
    }
    tc::tc_fence_before();
    __syncthreads();
    if (warp == kAdjWarps) {
        tc::tc_fence_after();
        tc::tmem_dealloc(tmem, tcols);
    }
}

int adj_nc(const Tab& t) { return (t.nin + t.nm + 15) / 16 * 16; }

}  // namespace

// The product's columns fit tensor memory (512), and a last block of them is at least 16 wide by rounding.
bool adjoint_fits(const Tab& t) { return adj_nc(t) <= 512 && t.nu % 2 == 0 && t.nin % 8 == 0; }

// FP32 in2out / in2sol of n elements from the solution columns of M (X, then Z), the residual R [n][nu][nin]
// and the angular sums of X.  err: device flag, set when a wait gave up.
elrt_status adjoint_correct(elrt_ctx* ctx, const float* M, int64_t ld, int64_t estride, const float* R, const void* sum,
                            float* in2out, float* in2sol, int* err, int64_t n) {
    const Tab& t = ctx->tab;
    AdjArgs g{};
    g.M = M;
    g.ld = ld;
    g.estride = estride;
    g.R = R;
    g.sum = (const ff*)sum;
    g.inv_n = ff_from_double_host(1.0 / t.N);
    g.jtiles = (t.nin + 127) / 128;
    g.jw = ((t.nin + g.jtiles - 1) / g.jtiles + 15) / 16 * 16;
    g.nc = adj_nc(t);
    g.stages = adj_smem(2, g.nc) <= kAdjSmem ? 2 : 1;
    g.err = err;
    const int smem = adj_smem(g.stages, g.nc);
    cudaError_t e = allow_smem(k_adjoint);
    if (e != cudaSuccess) return cuda_check(ctx, e, "smem attribute");
    ProfScope ps(ctx, "adjoint", 1,
                 (double)n * (t.nu * (2.0 * t.nin + t.nm) * 4.0 + t.nm * t.nin * 8.0 + (double)(t.nin + t.nm) * t.nin * 4.0),
                 2.0 * t.nu * (double)(t.nin + t.nm) * t.nin * n);
    k_adjoint<<<(unsigned)(n * g.jtiles), kAdjThreads, smem, ctx->stream>>>(t, g, in2out, in2sol);
    return cuda_check(ctx, cudaGetLastError(), "adjoint launch");
}
