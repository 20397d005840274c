// mlp.cu -- learned warm start: a 12 -> 64 -> 64 -> 64 -> 3 MLP (SiLU) that
// predicts a contact's converged impulse from local features, evaluated on
// the 5th-generation tensor cores (tcgen05: BF16 operands in shared memory,
// FP32 accumulators in TMEM) before the sweeps, and its training kernels
// (forward and backward on the tensor cores, Adam).
//
// Parameter layout (shared with every user of the network): for each layer
// the weight matrix W (out x in, row-major) then the bias b (out); 9,347
// FP32 values.
//
// Features of a contact (frame n, e2, e3 with e2 = -u_t/|u_t| along the
// free tangential relative velocity, or the contact frame's t when it is
// ~0; e3 = n x e2), all dimensionless:
//   0 u_n / v_ref            1 |u_t| / v_ref         2 (xi/dt) / v_ref
//   3..5 previous-step impulse (n, e2, e3) * w_n / v_ref
//   6 log(w_n)               7 w_t / w_n
//   8 r_a                    9 r_b (0 for a wall)
//   10 mu                    11 (contacts at j1 + contacts at j2) / 12
// u is the relative velocity of the free motion (velocities after the
// gravity kick, no contact impulses).  Output: the impulse in (n, e2, e3)
// times w_n / v_ref, computed as inputs 3..5 (the previous impulse) plus the
// network's correction; it is projected onto the friction cone.  It is used
// for contacts without a previous-step impulse; the others keep theirs (a
// converged previous impulse is far more accurate than any BF16 prediction
// where the contact network persists), as does a non-finite output.
#include <algorithm>
#include <cmath>

#include "mlp_tc.cuh"

namespace nbgs {

__device__ unsigned g_mlp_status;   // nbgs_mlp_infer: a tensor-core wait gave up

// --- plain inference on given rows (tests, evaluation) ------------------------
__global__ void __launch_bounds__(kTcRows) k_mlp_infer_tc(const float* __restrict__ theta, const float* __restrict__ X,
                                                          float* __restrict__ Y, int64_t n)
{
    extern __shared__ __align__(1024) unsigned char tc_smem[];
    TcMlpSmem& S = *reinterpret_cast<TcMlpSmem*>(tc_smem);
    tc_setup(theta, S);
    uint32_t phase = 0;
    bool ok = true;
    for (int64_t base = (int64_t)blockIdx.x * kTcRows; base < n; base += (int64_t)gridDim.x * kTcRows) {
        const int64_t row = base + threadIdx.x;
        float in[kIn], out[kOutN];
        if (row < n) {   // a row is 48 bytes: three 16-byte loads (X is 16-byte aligned)
            const float4* xr = reinterpret_cast<const float4*>(X + row * kIn);
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const float4 v = xr[q];
                in[4 * q] = v.x;
                in[4 * q + 1] = v.y;
                in[4 * q + 2] = v.z;
                in[4 * q + 3] = v.w;
            }
        } else {
#pragma unroll
            for (int k = 0; k < kIn; ++k) in[k] = 0.f;
        }
        if (ok && !tc_forward(S, in, out, phase)) {   // a wait gave up (uniform): NaN from here on
            ok = false;
            if (threadIdx.x == 0) atomicOr(&g_mlp_status, 1u);
        }
        if (row < n)   // skip connection: + previous impulse (inputs 3..5), in FP32
            for (int k = 0; k < kOutN; ++k) Y[row * kOutN + k] = ok ? out[k] + in[3 + k] : __int_as_float(0x7FC00000);
    }
    tc_teardown(S);
}

// --- training: forward and backward on the tensor cores (tcgen05) -----------
// One CTA per SM: two groups of 256 threads, each with a tile of 128 samples,
// and a warp whose first lane issues every MMA (so that the accumulations
// into the shared weight gradients stay in one thread's order).  Thread t of a
// group has sample t % 128 and columns 32 (t / 128) .. + 31 of each layer.  All
// products are tcgen05.mma with BF16 operands in shared memory (no swizzle)
// and FP32 accumulators in TMEM:
//   forward   Z_L   = A_{L-1} W_L^T        (M 128 samples, N out, K in)
//   backward  B_L   = D_L W_L              (M 128 samples, N in, K out)
//             dW_L += D_L^T A_{L-1}        (M out, padded to 128, N in, K 128 samples;
//                                           dW_4 transposed: its 16 columns instead of 64)
// with D_4 = (Y - T) / n, D_{L-1} = B_L * silu'(Z_{L-1} + b_{L-1}).  Every
// operand is stored once, in core matrices of 8 samples (or outputs) x 8
// features: a product that runs over features reads them as K-major, one that
// runs over samples or outputs as MN-major.  TMEM per group: two accumulators
// of 64 columns; Z_2 stays in one until the backward pass, silu'(Z_3) stays in
// registers and Z_1 is computed a second time.  The weight gradients
// accumulate in TMEM over all tiles of the CTA and are added to the global
// gradient once.  Bias gradients and the loss: FP32 sums of the unrounded
// deltas (a butterfly over the warp's samples leaves a column's sum in each
// lane, which keeps it for all tiles) and FP64.
//
// What bounds it is the exponential and the reciprocal of each sigmoid (five
// per hidden unit and sample, 16 such operations per clock and SM: 0.14 ms for
// 1M samples) and the eight hand-overs of a tile to the tensor cores, which the
// other group's tile hides in part.  1M samples: 325 us, against 2767 with
// one group of 128 threads, every operand stored in both orders and each
// column of the bias gradients reduced by itself.
constexpr int kTrRows = 128, kTrGroup = 256, kTrThreads = 2 * kTrGroup + 32;
constexpr int kTrCols = 512;                       // TMEM columns (one CTA per SM)
constexpr uint32_t kDW1 = 0, kDW2 = 16, kDW3 = 80, kDW4 = 144, kAcc = 160;   // TMEM column offsets; kAcc: 128 per group

struct TrainTile {
    alignas(128) __nv_bfloat16 a0[kTrRows * 16];           // inputs
    alignas(128) __nv_bfloat16 a[3][kTrRows * kHid];       // hidden activations
    alignas(128) __nv_bfloat16 d[kTrRows * kHid];          // deltas of the layer at hand
};
struct TrainTcSmem {
    TrainTile tile[2];   // a gradient's padding rows read up to 1 KB past an operand: what follows is defined memory
    alignas(128) __nv_bfloat16 w1[kHid * 16];              // W_L, rows = outputs, columns = inputs
    alignas(128) __nv_bfloat16 w2[kHid * kHid];
    alignas(128) __nv_bfloat16 w3[kHid * kHid];
    alignas(128) __nv_bfloat16 w4[16 * kHid];
    float b[3][kHid], b4[16];
    float gb[kHid * 3 + 16];                                // bias gradients b1, b2, b3, b4
    alignas(8) uint64_t ready[2], done[2];
    uint32_t tmem;
    int failed;
};

__device__ __forceinline__ void st_bf16(__nv_bfloat16* base, uint32_t byte_off, float v)
{
    *reinterpret_cast<__nv_bfloat16*>(reinterpret_cast<char*>(base) + byte_off) = __float2bfloat16_rn(v);
}

// Columns c0 .. c0 + 8 m of row r of an operand with K columns, 16 bytes a store.
template <int m>
__device__ __forceinline__ void st_cols(__nv_bfloat16* base, int r, int K, int c0, const float* v)
{
#pragma unroll
    for (int c = 0; c < 8 * m; c += 8) {
        const uint4 q = make_uint4(pack_bf16(v[c], v[c + 1]), pack_bf16(v[c + 2], v[c + 3]),
                                   pack_bf16(v[c + 4], v[c + 5]), pack_bf16(v[c + 6], v[c + 7]));
        *reinterpret_cast<uint4*>(reinterpret_cast<char*>(base) + kmaj_off(r, c0 + c, K)) = q;
    }
}

// 32 consecutive FP32 columns of this warp's 32 TMEM lanes (one row per thread).
__device__ __forceinline__ void tc_ld32(uint32_t taddr, float (&v)[32])
{
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
        "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]),
          "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
          "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]),
          "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int k = 0; k < 32; ++k) v[k] = __uint_as_float(r[k]);
}

// An operand of K_cols columns as the MMAs read it: over its columns (rows
// are the M or N index), or over its rows (its columns are).
struct TrOp {
    uint32_t addr, lbo, sbo, step;   // step: bytes from one MMA's 16 to the next
    int mn;
};
__device__ __forceinline__ TrOp over_cols(const void* p, int cols)
{
    return {smem_addr(p), 128u, (uint32_t)(cols / 8) * 128u, 256u, 0};
}
__device__ __forceinline__ TrOp over_rows(const void* p, int cols)
{
    const uint32_t lbo = (uint32_t)(cols / 8) * 128u;
    return {smem_addr(p), lbo, 128u, 2u * lbo, 1};
}

// K / 16 MMAs D(+)= A B^T of an M = 128 product; acc: accumulate into D from the first slice on.
__device__ __forceinline__ void tr_mma(uint32_t d, const TrOp& a, const TrOp& b, int K, int N, bool acc)
{
    const uint32_t idesc = tc_idesc(kTrRows, N) | ((uint32_t)a.mn << 15) | ((uint32_t)b.mn << 16);   // 1: MN-major
    for (int kk = 0; kk < K / 16; ++kk)
        tc_mma(d, tc_desc(a.addr + a.step * kk, a.lbo, a.sbo), tc_desc(b.addr + b.step * kk, b.lbo, b.sbo), idesc,
               (acc || kk > 0) ? 1 : 0);
}

// The eight hand-overs of a tile: what the tensor cores do with the operands
// that the group has just written.
__device__ __forceinline__ void tr_issue(TrainTcSmem& S, int step, int g, uint32_t tm, bool acc)
{
    TrainTile& t = S.tile[g];
    const uint32_t r0 = tm + kAcc + 128u * g, r1 = r0 + 64u;
    switch (step) {
    case 0: tr_mma(r0, over_cols(t.a0, 16), over_cols(S.w1, 16), 16, kHid, false); break;           // Z_1
    case 1: tr_mma(r1, over_cols(t.a[0], kHid), over_cols(S.w2, kHid), kHid, kHid, false); break;   // Z_2
    case 2: tr_mma(r0, over_cols(t.a[1], kHid), over_cols(S.w3, kHid), kHid, kHid, false); break;   // Z_3
    case 3: tr_mma(r0, over_cols(t.a[2], kHid), over_cols(S.w4, kHid), kHid, 16, false); break;     // Z_4
    case 4:
        tr_mma(r0, over_cols(t.d, 16), over_rows(S.w4, kHid), 16, kHid, false);                     // B_4
        tr_mma(tm + kDW4, over_rows(t.a[2], kHid), over_rows(t.d, 16), kTrRows, 16, acc);
        break;
    case 5:
        tr_mma(r0, over_cols(t.d, kHid), over_rows(S.w3, kHid), kHid, kHid, false);                 // B_3
        tr_mma(tm + kDW3, over_rows(t.d, kHid), over_rows(t.a[1], kHid), kTrRows, kHid, acc);
        break;
    case 6:
        tr_mma(r0, over_cols(t.d, kHid), over_rows(S.w2, kHid), kHid, kHid, false);                 // B_2
        tr_mma(r1, over_cols(t.a0, 16), over_cols(S.w1, 16), 16, kHid, false);                      // Z_1 again
        tr_mma(tm + kDW2, over_rows(t.d, kHid), over_rows(t.a[0], kHid), kTrRows, kHid, acc);
        break;
    default: tr_mma(tm + kDW1, over_rows(t.d, kHid), over_rows(t.a0, 16), kTrRows, 16, acc); break;
    }
}

// Operands written and accumulators read -> the issuing warp; then wait for
// its MMAs.  False when the wait gave up.
__device__ __forceinline__ bool tr_step(TrainTcSmem& S, int g, uint32_t& phase)
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(&S.ready[g])) : "memory");
    const bool ok = tc_wait(&S.done[g], phase & 1u);
    phase += 1u;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    return __all_sync(0xffffffffu, ok) != 0;   // a warp stays together
}

// 1 / (1 + e^-z): the hardware's approximate reciprocal (within one unit in the
// last place) and one step of the Newton-Raphson iteration y (2 - d y), after
// which the error is that of the last rounding (tests/test_reciprocal_method.py).
// z from -80 on: the step wants a finite denominator, and what is below is 1e-35
// either way.  The library's __frcp_rn, with its branch: 1M samples 543 us, 342 this way.
__device__ __forceinline__ float sigmoid_f(float z)
{
    const float d = 1.f + __expf(-fmaxf(z, -80.f));
    float y;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(d));
    return fmaf(fmaf(-d, y, 1.f), y, y);
}
__device__ __forceinline__ float silu_grad_f(float z, float sg) { return sg * (1.f + z * (1.f - sg)); }

// Sum over the warp's lanes (samples) of v[0..31] (columns): column `lane`'s. v is used up.
__device__ __forceinline__ float column_sum(float (&v)[32])
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        const bool up = (threadIdx.x & o) != 0u;
#pragma unroll
        for (int k = 0; k < o; ++k) {
            const float give = up ? v[k] : v[k + o], keep = up ? v[k + o] : v[k];
            v[k] = keep + __shfl_xor_sync(0xffffffffu, give, o);
        }
    }
    return v[0];
}

__global__ void __launch_bounds__(kTrThreads, 1) k_mlp_grad_tc(const float* __restrict__ th, const float* __restrict__ X,
                                                            const float* __restrict__ T, int64_t n,
                                                            float* __restrict__ grad, double* __restrict__ loss,
                                                            unsigned* status)
{
    extern __shared__ __align__(1024) unsigned char tr_smem[];
    TrainTcSmem& S = *reinterpret_cast<TrainTcSmem*>(tr_smem);
    const int tid = threadIdx.x, lane = tid & 31;
    // weights, biases, bias gradients; the tiles start from zeros (the
    // gradients' padding rows read them before they are written)
    for (int e = tid; e < (int)(sizeof(S.tile) / 16); e += kTrThreads)
        reinterpret_cast<uint4*>(S.tile)[e] = make_uint4(0u, 0u, 0u, 0u);
    for (int e = tid; e < kHid * 16; e += kTrThreads) {
        const int o = e / 16, i = e % 16;
        st_bf16(S.w1, kmaj_off(o, i, 16), i < kIn ? th[kOffW1 + o * kIn + i] : 0.f);
    }
    for (int e = tid; e < kHid * kHid; e += kTrThreads) {
        const int o = e / kHid, i = e % kHid;
        st_bf16(S.w2, kmaj_off(o, i, kHid), th[kOffW2 + o * kHid + i]);
        st_bf16(S.w3, kmaj_off(o, i, kHid), th[kOffW3 + o * kHid + i]);
    }
    for (int e = tid; e < 16 * kHid; e += kTrThreads) {
        const int o = e / kHid, i = e % kHid;
        st_bf16(S.w4, kmaj_off(o, i, kHid), o < kOutN ? th[kOffW4 + o * kHid + i] : 0.f);
    }
    for (int k = tid; k < kHid; k += kTrThreads) {
        S.b[0][k] = th[kOffB1 + k];
        S.b[1][k] = th[kOffB2 + k];
        S.b[2][k] = th[kOffB3 + k];
    }
    if (tid < 16) S.b4[tid] = tid < kOutN ? th[kOffB4 + tid] : 0.f;
    for (int k = tid; k < kHid * 3 + 16; k += kTrThreads) S.gb[k] = 0.f;
    if (tid == 0) {
        for (int g = 0; g < 2; ++g) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(&S.ready[g])), "r"(kTrGroup) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&S.done[g])) : "memory");
        }
        S.failed = 0;
    }
    if (tid < 32) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&S.tmem)),
                     "r"(kTrCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // weights: generic stores -> MMA reads
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tm = S.tmem;
    // tiles of this CTA's groups: 2 b + g, then every 2 gridDim.x
    const int64_t tiles = (n + kTrRows - 1) / kTrRows, tstride = 2 * (int64_t)gridDim.x;
    if (tid == 2 * kTrGroup) {   // the issuing lane
        int64_t left[2];
        for (int g = 0; g < 2; ++g) left[g] = (tiles - (2 * (int64_t)blockIdx.x + g) + tstride - 1) / tstride;
        uint32_t phase = 0;
        uint32_t begun = 0;   // steps whose gradient has been started
        bool ok = true;
        for (int64_t k = 0; ok && (k < left[0] || k < left[1]); ++k) {
            for (int step = 0; step < 8 && ok; ++step, ++phase) {
                for (int g = 0; g < 2 && ok; ++g) {
                    if (k >= left[g]) continue;
                    ok = tc_wait(&S.ready[g], phase & 1u);
                    if (!ok) break;
                    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                    tr_issue(S, step, g, tm, (begun >> step & 1u) != 0u);
                    begun |= 1u << step;
                    tc_commit(&S.done[g]);
                }
            }
        }
        if (!ok) S.failed = 1;
    } else if (tid < 2 * kTrGroup) {
        const int g = tid / kTrGroup, r = tid & (kTrRows - 1), h = (tid / kTrRows) & 1, c0 = 32 * h;
        TrainTile& A = S.tile[g];
        const uint32_t r0 = tm + ((uint32_t)(r & ~31) << 16) + kAcc + 128u * g, r1 = r0 + 64u;
        const float inv_n = 1.f / (float)n;
        const bool wide = ((uintptr_t)X & 15u) == 0u;
        double lsum = 0.0;
        float gb1 = 0.f, gb2 = 0.f, gb3 = 0.f, gb4[kOutN] = {0.f, 0.f, 0.f};
        uint32_t phase = 0;
        bool ok = true;
        auto bias4 = [&](int L, int k) { return *reinterpret_cast<const float4*>(&S.b[L][c0 + k]); };
        // a hidden layer's activations from its accumulator; its derivative if asked
        float v[32], g3[32];
        auto hidden = [&](uint32_t acc, int L, bool keep) {
            tc_ld32(acc + c0, v);
#pragma unroll
            for (int k = 0; k < 32; k += 4) {
                const float4 b = bias4(L, k);
                const float z[4] = {v[k] + b.x, v[k + 1] + b.y, v[k + 2] + b.z, v[k + 3] + b.w};
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                    const float sg = sigmoid_f(z[q]);
                    if (keep) g3[k + q] = silu_grad_f(z[q], sg);
                    v[k + q] = z[q] * sg;
                }
            }
            st_cols<4>(A.a[L], r, kHid, c0, v);
        };
        // a hidden layer's deltas from B in r0 and its pre-activations in r1
        auto deltas = [&](int L) {
            float z[32];
            tc_ld32(r1 + c0, z);
#pragma unroll
            for (int k = 0; k < 32; k += 4) {
                const float4 b = bias4(L, k);
                const float zz[4] = {z[k] + b.x, z[k + 1] + b.y, z[k + 2] + b.z, z[k + 3] + b.w};
#pragma unroll
                for (int q = 0; q < 4; ++q) z[k + q] = silu_grad_f(zz[q], sigmoid_f(zz[q]));
            }
            tc_ld32(r0 + c0, v);
#pragma unroll
            for (int k = 0; k < 32; ++k) v[k] *= z[k];
            st_cols<4>(A.d, r, kHid, c0, v);
        };
        for (int64_t tile = 2 * (int64_t)blockIdx.x + g; tile < tiles; tile += tstride) {
            const int64_t row = tile * kTrRows + r;
            const bool valid = row < n;
            float x[8], t[kOutN];
#pragma unroll
            for (int k = 0; k < 8; ++k) x[k] = 0.f;
            if (valid) {
                const float* xr = X + row * kIn + 8 * h;   // inputs 0 .. 7 or 8 .. 11
                if (wide) {
                    const float4 p = *reinterpret_cast<const float4*>(xr);
                    x[0] = p.x;
                    x[1] = p.y;
                    x[2] = p.z;
                    x[3] = p.w;
                    if (h == 0) {
                        const float4 q = *reinterpret_cast<const float4*>(xr + 4);
                        x[4] = q.x;
                        x[5] = q.y;
                        x[6] = q.z;
                        x[7] = q.w;
                    }
                } else {
#pragma unroll
                    for (int k = 0; k < 8; ++k)
                        if (k < 4 || h == 0) x[k] = xr[k];
                }
            }
#pragma unroll
            for (int k = 0; k < kOutN; ++k) t[k] = valid && h == 0 ? T[row * kOutN + k] : 0.f;
            st_cols<1>(A.a0, r, 16, 8 * h, x);
            if (!(ok = tr_step(S, g, phase))) break;
            hidden(r0, 0, false);
            if (!(ok = tr_step(S, g, phase))) break;
            hidden(r1, 1, false);
            if (!(ok = tr_step(S, g, phase))) break;
            hidden(r0, 2, true);
            if (!(ok = tr_step(S, g, phase))) break;
            // output, loss, D_4
            {
                float d4[8];
#pragma unroll
                for (int k = 0; k < 8; ++k) d4[k] = 0.f;
                if (h == 0) {
                    float y[16];
                    tc_ld16(r0, y);
#pragma unroll
                    for (int k = 0; k < kOutN; ++k) {
                        const float e = valid ? (y[k] + S.b4[k] + x[3 + k]) - t[k] : 0.f;
                        lsum = fma((double)e, (double)e, lsum);
                        d4[k] = e * inv_n;
                        gb4[k] += d4[k];
                    }
                }
                st_cols<1>(A.d, r, 16, 8 * h, d4);
            }
            if (!(ok = tr_step(S, g, phase))) break;
            tc_ld32(r0 + c0, v);
#pragma unroll
            for (int k = 0; k < 32; ++k) v[k] *= g3[k];
            st_cols<4>(A.d, r, kHid, c0, v);
            gb3 += column_sum(v);
            if (!(ok = tr_step(S, g, phase))) break;
            deltas(1);
            gb2 += column_sum(v);
            if (!(ok = tr_step(S, g, phase))) break;
            deltas(0);
            gb1 += column_sum(v);
            if (!(ok = tr_step(S, g, phase))) break;
        }
        if (!ok) S.failed = 1;
        atomicAdd(&S.gb[c0 + lane], gb1);
        atomicAdd(&S.gb[kHid + c0 + lane], gb2);
        atomicAdd(&S.gb[2 * kHid + c0 + lane], gb3);
        if (h == 0) {
#pragma unroll
            for (int k = 0; k < kOutN; ++k) {
                float q = gb4[k];
                for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
                if (lane == 0) atomicAdd(&S.gb[3 * kHid + k], q);
            }
            for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
            if (lane == 0 && lsum != 0.0) atomicAdd(loss, 0.5 * lsum / (double)n);
        }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const bool ok = S.failed == 0;
    if (!ok && tid == 0) atomicOr(status, 1u);
    // The gradients: rows 0 .. 63 of the TMEM accumulators (warps 0 and 1 of
    // each four), through shared memory in the parameters' order, so that the
    // atomics of a warp fall on neighbouring addresses.
    float* const out = reinterpret_cast<float*>(S.tile);
    if (ok && tid < 2 * kTrGroup && (tid & (kTrRows - 1)) < kHid) {
        const int r = tid & (kTrRows - 1), part = tid / kTrRows;
        const uint32_t ln = (uint32_t)(r & ~31) << 16;
        float v[32];
        tc_ld32(tm + ln + kDW2 + 32u * part, v);   // dW_2 and dW_3: 128 columns, 32 for each of four
        float* o = out + (part < 2 ? kOffW2 : kOffW3) + r * kHid + 32 * (part & 1);
#pragma unroll
        for (int k = 0; k < 32; ++k) o[k] = v[k];
        if (part < 2) {
            float w[16];
            tc_ld16(tm + ln + (part == 0 ? kDW1 : kDW4), w);
            if (part == 0) {
#pragma unroll
                for (int k = 0; k < kIn; ++k) out[kOffW1 + r * kIn + k] = w[k];
            } else {
#pragma unroll
                for (int k = 0; k < kOutN; ++k) out[kOffW4 + k * kHid + r] = w[k];
            }
        }
    }
    for (int k = tid; k < kHid * 3 + kOutN; k += kTrThreads)
        out[(k < kHid ? kOffB1 : k < 2 * kHid ? kOffB2 : k < 3 * kHid ? kOffB3 : kOffB4) + k % kHid] = S.gb[k];
    __syncthreads();
    if (ok)
        for (int k = tid; k < kNParams; k += kTrThreads) atomicAdd(&grad[k], out[k]);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (tid < 32) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tm), "r"(kTrCols) : "memory");
    }
}

__global__ void k_adam(float* __restrict__ th, const float* __restrict__ g, float* __restrict__ m, float* __restrict__ v,
                       int64_t count, float lr, float b1, float b2, float eps, float c1, float c2)
{
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < count; k += (int64_t)gridDim.x * blockDim.x) {
        const float gk = g[k];
        const float mk = b1 * m[k] + (1.f - b1) * gk;
        const float vk = b2 * v[k] + (1.f - b2) * gk * gk;
        m[k] = mk;
        v[k] = vk;
        th[k] -= lr * (mk / c1) / (sqrtf(vk / c2) + eps);
    }
}

// One CTA: 128 contacts per tile (warm_tiles).
template <class R>
__global__ void __launch_bounds__(kTcRows) k_mlp_warmstart(WarmArgs<R> A)
{
    extern __shared__ __align__(1024) unsigned char tc_smem[];
    warm_tiles<R>(A, A.apply ? reinterpret_cast<TcMlpSmem*>(tc_smem) : nullptr);
}

// Features (and, with apply, the network's warm start) for the current
// contacts; runs before the sweeps (after colouring, before the gravity kick).
nbgs_status run_mlp_prologue(nbgs_scene* s, int apply, float* feat_out)
{
    if (s->composite) return fail(s, NBGS_EINVAL, "MLP: the network takes sphere contacts only");
    const int64_t C = s->n_contacts;
    if (C <= 0) return NBGS_OK;
    if (apply && !s->mlp_theta) return fail(s, NBGS_EINVAL, "MLP warm start: no network loaded (nbgs_mlp_load)");
    const int gb = grid_for(C, kTcRows, 4, s->num_sms);
    const size_t smem = apply ? sizeof(TcMlpSmem) : 0;
    if (s->fp32) k_mlp_warmstart<float><<<gb, kTcRows, smem, s->stream>>>(warm_args<float>(s, apply, feat_out));
    else k_mlp_warmstart<double><<<gb, kTcRows, smem, s->stream>>>(warm_args<double>(s, apply, feat_out));
    if (s->timing) s->phase_launches[2] += 1;
    return cuda_check(s, cudaGetLastError(), "MLP prologue");
}

}  // namespace nbgs

using namespace nbgs;

extern "C" {

nbgs_status nbgs_mlp_infer(const float* theta, const float* X, float* Y, int64_t n, void* stream)
{
    if (!theta || n < 0 || (n > 0 && (!X || !Y)) || ((uintptr_t)X & 15u)) return NBGS_EINVAL;
    if (n == 0) return NBGS_OK;
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t tiles = (n + kTcRows - 1) / kTcRows;
    k_mlp_infer_tc<<<grid_for(tiles * kTcRows, kTcRows, 4, sms), kTcRows, sizeof(TcMlpSmem), (cudaStream_t)stream>>>(
        theta, X, Y, n);
    return cudaGetLastError() == cudaSuccess ? NBGS_OK : NBGS_ECUDA;
}

nbgs_status nbgs_mlp_grad(const float* theta, const float* X, const float* T, int64_t n, float* grad, double* loss,
                          void* stream)
{
    if (!theta || !grad || !loss || n <= 0 || !X || !T) return NBGS_EINVAL;
    cudaStream_t st = (cudaStream_t)stream;
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    static_assert(sizeof(TrainTcSmem) < 227 * 1024, "training tile too large");
    const int smem = (int)sizeof(TrainTcSmem);
    if (cudaFuncSetAttribute(k_mlp_grad_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, smem) != cudaSuccess)
        return NBGS_ECUDA;
    unsigned* status = nullptr;
    if (cudaGetSymbolAddress((void**)&status, g_mlp_status) != cudaSuccess) return NBGS_ECUDA;
    cudaMemsetAsync(grad, 0, kNParams * sizeof(float), st);
    cudaMemsetAsync(loss, 0, sizeof(double), st);
    const int64_t pairs = ((n + kTrRows - 1) / kTrRows + 1) / 2;      // two tiles at a time
    const int blocks = (int)std::min<int64_t>(pairs, (int64_t)sms);   // one CTA per SM (all of its TMEM)
    k_mlp_grad_tc<<<blocks, kTrThreads, smem, st>>>(theta, X, T, n, grad, loss, status);
    return cudaGetLastError() == cudaSuccess ? NBGS_OK : NBGS_ECUDA;
}

nbgs_status nbgs_mlp_adam(float* theta, const float* grad, float* m, float* v, int64_t count, float lr, float beta1,
                          float beta2, float eps, int32_t step, void* stream)
{
    if (!theta || !grad || !m || !v || count <= 0 || step < 1) return NBGS_EINVAL;
    const float c1 = 1.f - powf(beta1, (float)step), c2 = 1.f - powf(beta2, (float)step);
    k_adam<<<(int)((count + 255) / 256), 256, 0, (cudaStream_t)stream>>>(theta, grad, m, v, count, lr, beta1, beta2, eps,
                                                                        c1, c2);
    return cudaGetLastError() == cudaSuccess ? NBGS_OK : NBGS_ECUDA;
}

nbgs_status nbgs_mlp_load(nbgs_scene* s, const float* theta, int64_t count)
{
    NBGS_GUARD(s);
    if (!theta || count != kNParams) return fail(s, NBGS_EINVAL, "mlp_load: expected 9347 parameters");
    if (!s->mlp_theta) {
        s->mlp_theta = (float*)dev_alloc(s, kNParams * sizeof(float));
        if (!s->mlp_theta) return fail(s, NBGS_ENOMEM, "mlp_load: allocation");
    }
    return cuda_check(s, cudaMemcpyAsync(s->mlp_theta, theta, kNParams * sizeof(float), cudaMemcpyDefault, s->stream),
                      "mlp_load");
}

nbgs_status nbgs_mlp_features(nbgs_scene* s, float* out, int64_t cap, int64_t* n_out)
{
    NBGS_GUARD(s);
    if (!s->coloured) return fail(s, NBGS_EINVAL, "mlp_features: detect and colour the contacts first");
    if (n_out) *n_out = s->n_contacts;
    if (!out || cap < s->n_contacts || s->n_contacts == 0) return NBGS_OK;
    float* buf = (float*)dev_alloc(s, (size_t)s->n_contacts * 16 * sizeof(float));
    if (!buf) return fail(s, NBGS_ENOMEM, "mlp_features: staging");
    nbgs_status rc = run_mlp_prologue(s, 0, buf);
    if (rc == NBGS_OK)
        rc = cuda_check(s, cudaMemcpyAsync(out, buf, (size_t)s->n_contacts * 16 * sizeof(float), cudaMemcpyDefault,
                                           s->stream), "mlp_features");
    if (rc == NBGS_OK) rc = cuda_check(s, cudaStreamSynchronize(s->stream), "mlp_features");
    dev_free(s, buf);
    return rc;
}

}  // extern "C"
