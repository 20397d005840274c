// relax.cuh -- the relaxation of one sphere contact (Sect. 3, Sect. 5
// Alg. 1), shared by the sweep kernels: record decoding and the arithmetic on
// loaded bodies.
#pragma once

#include "nbgs_internal.cuh"

namespace nbgs {

template <class R>
__device__ __forceinline__ void decode(const SweepRec<R>& r, uint32_t& a, uint32_t& b, R& la, R& lb, R& nx, R& ny, R& nz,
                                       R& bias);

template <>
__device__ __forceinline__ void decode<float>(const SweepRec<float>& r, uint32_t& a, uint32_t& b, float& la, float& lb,
                                              float& nx, float& ny, float& nz, float& bias)
{
    a = __float_as_uint(r.a.x);
    b = __float_as_uint(r.a.y);
    la = r.a.z;
    lb = r.a.w;
    nx = r.b.x;
    ny = r.b.y;
    nz = r.b.z;
    bias = r.b.w;
}

template <>
__device__ __forceinline__ void decode<double>(const SweepRec<double>& r, uint32_t& a, uint32_t& b, double& la,
                                               double& lb, double& nx, double& ny, double& nz, double& bias)
{
    const uint64_t ids = (uint64_t)__double_as_longlong(r.ids_bias.x);
    a = (uint32_t)(ids & 0xFFFFFFFFu);
    b = (uint32_t)(ids >> 32);
    bias = r.ids_bias.y;
    la = r.lev.x;
    lb = r.lev.y;
    nx = r.nxy.x;
    ny = r.nxy.y;
    nz = r.nz_.x;
}

// Sweep records do not change during a solve.
__device__ __forceinline__ SweepRec<float> ld_rec(const SweepRec<float>* p)
{
    SweepRec<float> r;
    asm("ld.global.nc.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
        : "=f"(r.a.x), "=f"(r.a.y), "=f"(r.a.z), "=f"(r.a.w), "=f"(r.b.x), "=f"(r.b.y), "=f"(r.b.z), "=f"(r.b.w)
        : "l"(p));
    return r;
}
__device__ __forceinline__ SweepRec<double> ld_rec(const SweepRec<double>* p)
{
    SweepRec<double> r;
    asm("ld.global.nc.v4.f64 {%0,%1,%2,%3}, [%4];"
        : "=d"(r.ids_bias.x), "=d"(r.ids_bias.y), "=d"(r.lev.x), "=d"(r.lev.y)
        : "l"(p));
    asm("ld.global.nc.v4.f64 {%0,%1,%2,%3}, [%4];"
        : "=d"(r.nxy.x), "=d"(r.nxy.y), "=d"(r.nz_.x), "=d"(r.nz_.y)
        : "l"(reinterpret_cast<const char*>(p) + 32));
    return r;
}

// State of the two bodies of a contact: (v, 1/m), (w, 1/I) each.
template <class R> struct Bodies {
    R4<R> va, wa, vb, wb;
};

// omega y + (1 - omega) p.  FP32: the operations fused one way, written out,
// because the compiler fuses a plain expression differently from one kernel to
// the next, and every schedule of the sweeps gives the same bits.
__device__ __forceinline__ float blend(float omega, float y, float om1, float p)
{
    return fmaf(om1, p, __fmul_rn(omega, y));
}
__device__ __forceinline__ double blend(double omega, double y, double om1, double p) { return omega * y + om1 * p; }


// Relax one contact (apply_only: add its stored impulse instead) on loaded
// bodies: the impulse p (xyz) and the velocities in B are updated, and r_j^2
// = |W (p_new - p_old)|^2 is returned.  False in `moves` when both masses are
// infinite: nothing changes.  The square root of r_j^2 is left to the caller
// (it is monotone, so the largest r_j is the root of the largest r_j^2).
template <class R, bool apply_only>
__device__ __forceinline__ R relax_bodies(const SweepRec<R>& rr, R mu, R omega, R4<R>& pp, Bodies<R>& B, bool& moves)
{
    uint32_t ia, ib;
    R la, lb, nx, ny, nz, bias;
    decode<R>(rr, ia, ib, la, lb, nx, ny, nz, bias);
    R4<R>&va = B.va, &wa = B.wa, &vb = B.vb, &wb = B.wb;
    const R ima = va.w, iIa = wa.w, imb = vb.w, iIb = wb.w;
    R tx, ty, tz, ox, oy, oz;
    tangent_basis<R>(nx, ny, nz, tx, ty, tz, ox, oy, oz);
    const R wn = ima + imb;
    moves = wn > R(0);
    if (!moves) return R(0);
    const R wt = wn + iIa * la * la + iIb * lb * lb;
    R dn, dt_, do_;
    if (apply_only) {
        dn = pp.x;
        dt_ = pp.y;
        do_ = pp.z;
    } else {
        // u = v_a - la (w_a x n) - v_b - lb (w_b x n)
        const R cax = wa.y * nz - wa.z * ny, cay = wa.z * nx - wa.x * nz, caz = wa.x * ny - wa.y * nx;
        const R cbx = wb.y * nz - wb.z * ny, cby = wb.z * nx - wb.x * nz, cbz = wb.x * ny - wb.y * nx;
        const R ux = (va.x - la * cax) - (vb.x + lb * cbx);
        const R uy = (va.y - la * cay) - (vb.y + lb * cby);
        const R uz = (va.z - la * caz) - (vb.z + lb * cbz);
        const R un = nx * ux + ny * uy + nz * uz;
        const R ut = tx * ux + ty * uy + tz * uz;
        const R uo = ox * ux + oy * uy + oz * uz;
        const R bn = un - wn * pp.x + bias;
        const R bt = ut - wt * pp.y;
        const R bo = uo - wt * pp.z;
        R yn = -bn / wn;
        yn = yn > R(0) ? yn : R(0);
        R yt = -bt / wt, yo = -bo / wt;
        const R lim = mu * yn;
        const R len2 = yt * yt + yo * yo;
        if (len2 > lim * lim) {
            if (len2 > R(0)) {
                const R sc = lim / sqrt(len2);
                yt *= sc;
                yo *= sc;
            } else {
                yt = yo = R(0);
            }
        }
        const R om1 = R(1) - omega;
        const R pn = blend(omega, yn, om1, pp.x), pt = blend(omega, yt, om1, pp.y), po = blend(omega, yo, om1, pp.z);
        dn = pn - pp.x;
        dt_ = pt - pp.y;
        do_ = po - pp.z;
        pp.x = pn;
        pp.y = pt;
        pp.z = po;
    }
    // world impulse change P = dn n + dt t + do o; torque arm n x P
    const R Px = dn * nx + dt_ * tx + do_ * ox;
    const R Py = dn * ny + dt_ * ty + do_ * oy;
    const R Pz = dn * nz + dt_ * tz + do_ * oz;
    const R qx = ny * Pz - nz * Py, qy = nz * Px - nx * Pz, qz = nx * Py - ny * Px;
    if (ima > R(0) || iIa > R(0)) {
        va.x += ima * Px;
        va.y += ima * Py;
        va.z += ima * Pz;
        const R ka = la * iIa;
        wa.x -= ka * qx;
        wa.y -= ka * qy;
        wa.z -= ka * qz;
    }
    if (imb > R(0) || iIb > R(0)) {
        vb.x -= imb * Px;
        vb.y -= imb * Py;
        vb.z -= imb * Pz;
        const R kb = lb * iIb;
        wb.x -= kb * qx;
        wb.y -= kb * qy;
        wb.z -= kb * qz;
    }
    const R r1 = wn * dn, r2 = wt * dt_, r3 = wt * do_;
    return r1 * r1 + r2 * r2 + r3 * r3;
}

// --- pieces of the relaxation on several lanes (units.cuh) -------------------
// x / w from the reciprocal y of w rounded to nearest: the remainder x - w q
// of q = x y is exact in one fused multiply-add, and RN(q + (x - w q) y) is
// the correctly rounded quotient (Markstein's theorem, as in the detection's
// normals): three operations instead of a division.  For w in the range of
// recip_ok.
template <class R>
__device__ __forceinline__ R quotient(R x, R w, R y)
{
    const R q = x * y;
    return fma(fma(-q, w, x), y, q);
}
__device__ __forceinline__ bool recip_ok(float wn, float wt) { return wn > 1e-30f && wt < 1e30f; }   // wn <= wt
__device__ __forceinline__ bool recip_ok(double wn, double wt) { return wn > 1e-250 && wt < 1e250; }

// a > b for a, b >= 0 or NaN-free of sign: FP64 compares on their bits (the
// FP64 unit takes 64 cycles for any instruction of a warp, an integer compare
// a few).
__device__ __forceinline__ bool above(float a, float b) { return a > b; }
__device__ __forceinline__ bool above(double a, double b) { return __double_as_longlong(a) > __double_as_longlong(b); }
// a > b for a >= 0 and b >= 0 or NaN, of either sign: nothing is above a NaN (the
// limit of a separating contact under an infinite friction coefficient).
__device__ __forceinline__ bool beyond(double a, double b)
{
    return (unsigned long long)__double_as_longlong(a) > (unsigned long long)__double_as_longlong(b);
}
// max(0, y), 0 for NaN
__device__ __forceinline__ float clamp0(float y) { return y > 0.f ? y : 0.f; }
__device__ __forceinline__ double clamp0(double y)
{
    const long long b = __double_as_longlong(y);
    return b > 0 && b <= 0x7FF0000000000000LL ? y : 0.0;
}

// lim / sqrt(len2) for len2 > lim^2 >= 0 in FP64, by the library's reciprocal
// square root (within one unit in the last place).  A step of 1,000 spheres: 1,859
// us, 1,936 with the hardware's approximation refined by hand.
__device__ __forceinline__ double slide_scale(double lim, double len2) { return lim * rsqrt(len2); }

template <class R>
__device__ __forceinline__ double block_max_to(R v, unsigned long long* dst)
{
    __shared__ double sm[32];
    double x = (double)v;
    for (int o = 16; o > 0; o >>= 1) x = fmax(x, __shfl_down_sync(0xffffffffu, x, o));
    if ((threadIdx.x & 31) == 0) sm[threadIdx.x >> 5] = x;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < (int)(blockDim.x >> 5); ++k) x = fmax(x, sm[k]);
        if (!(x <= 1e300)) x = __longlong_as_double(0x7FF0000000000000LL);  // NaN/Inf -> +Inf
        atomicMax(dst, (unsigned long long)__double_as_longlong(x));
    }
    __syncthreads();
    return x;
}

__device__ __forceinline__ double v_ref_of(const DevInfo* info, double gdt_norm)
{
    double v = __longlong_as_double((long long)info->vmax_bits);
    v = fmax(v, gdt_norm);
    return fmax(v, 1e-12);
}

// --- TMA bulk copies (global -> shared) completed on an mbarrier -----------
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t* bar)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(bar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* bar)
{
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar)) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile("{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
                 "selp.u32 %0, 1, 0, p;\n\t}"
                 : "=r"(ok) : "r"(smem_u32(bar)), "r"(parity) : "memory");
    return ok != 0;
}

// Bounded wait for the stage of the given parity; false (timeout bit set)
// after ~2^31 SM clocks.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, DevInfo* info)
{
    const long long t0 = clock64();
    while (!mbar_try_wait(bar, parity)) {
        if (clock64() - t0 > (1LL << 31)) {
            atomicOr(&info->err, kErrTimeout);
            return false;
        }
    }
    return true;
}

// One end of a contact's dependency word from the colours of its body's
// contacts (mask, 256 bits): the colour below c and whether c is the highest.
__device__ __forceinline__ uint32_t dep_end(const uint32_t* __restrict__ mask, uint32_t c)
{
    const uint4* q = reinterpret_cast<const uint4*>(mask);
    const uint4 lo = q[0], hi = q[1];
    const uint32_t m[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
    const uint32_t wd = c >> 5, bit = c & 31u;
    uint32_t pred = 0u;
    bool last = true;
#pragma unroll
    for (uint32_t k = 0; k < 8; ++k) {
        const uint32_t below = k < wd ? m[k] : (k == wd ? m[k] & ((1u << bit) - 1u) : 0u);
        const uint32_t above = k > wd ? m[k] : (k == wd ? (m[k] >> bit) >> 1 : 0u);
        if (below) pred = 32u * k + 32u - (uint32_t)__clz((int)below);   // colour + 1
        if (above) last = false;
    }
    return pred | (last ? kDepLastA : 0u) | kDepListA;
}

// Rotating per-scene residual slot of sweep k (three, so that clearing the
// slot of sweep k + 1 while sweep k runs touches nothing still read).
__host__ __device__ __forceinline__ int scene_slot(int k) { return k % 3; }

// The tolerance test of sweep k without a grid barrier.  R_k <= tol holds
// exactly when every block's own maximum (divided by the same v_ref) is at
// or below tol, so a block above it announces that and goes on at once; a
// block at or below it counts itself and waits until either some block has
// announced (the sweeps go on) or every block has counted itself (the solve
// stops after sweep k).  Every block reaches the end of sweep k, so the
// wait ends; bounded like every other.  Returns 1 to go on, 0 to stop, -1
// when the wait ran out.
__device__ __forceinline__ int tol_vote(DevInfo* info, int k, double rb, double vnorm, double tol, unsigned nb,
                                        int* s_vote)
{
    if (threadIdx.x == 0) {
        uint32_t* flag = info->votes + 2 * k;
        int v = 1;
        if (!(rb / vnorm <= tol)) {
            if (((volatile uint32_t*)flag)[0] == 0u) atomicExch(flag, 1u);
        } else {
            atomicAdd(flag + 1, 1u);
            const long long t0 = clock64();
            for (;;) {
                if (((volatile uint32_t*)flag)[0] != 0u) break;
                if (((volatile uint32_t*)flag)[1] == nb) {
                    v = 0;
                    break;
                }
                if ((((volatile uint32_t*)&info->err)[0] & kErrTimeout) || clock64() - t0 > (1LL << 31)) {
                    atomicOr(&info->err, kErrTimeout);
                    v = -1;
                    break;
                }
            }
        }
        *s_vote = v;
    }
    __syncthreads();
    return *s_vote;
}

}  // namespace nbgs
