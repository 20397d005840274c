// integrate.cu -- time integration (Sect. 3, eq. integrationscheme) and the
// conversions between the caller's double arrays and the body layout.
#include <cstring>

#include "nbgs_internal.cuh"

namespace nbgs {

// An FP64 instruction, conversions and comparisons among them, occupies a
// scheduler's FP64 unit for 64 cycles.  Conversions of numbers that are exact
// in both formats are moves of their fields; others (subnormal, not finite, or
// with bits that FP32 does not hold) take the instruction.
__device__ __forceinline__ double widen(float f)
{
    const uint32_t b = __float_as_uint(f), m = b & 0x7FFFFFFFu, sign = b & 0x80000000u;
    if (m - 0x00800000u < 0x7F000000u) return __hiloint2double((int)(sign | ((m >> 3) + 0x38000000u)), (int)(b << 29));
    if (m == 0u) return __hiloint2double((int)sign, 0);
    return (double)f;
}
__device__ __forceinline__ double widen(double x) { return x; }
template <class R> __device__ __forceinline__ R narrow_to(double x);
template <> __device__ __forceinline__ double narrow_to<double>(double x) { return x; }
template <> __device__ __forceinline__ float narrow_to<float>(double x)
{
    const uint32_t hi = (uint32_t)__double2hiint(x), lo = (uint32_t)__double2loint(x), m = hi & 0x7FFFFFFFu;
    if ((lo & 0x1FFFFFFFu) == 0u) {
        if (m - 0x38100000u < 0x47F00000u - 0x38100000u)
            return __uint_as_float((hi & 0x80000000u) | ((m - 0x38000000u) << 3) | (lo >> 29));
        if ((m | lo) == 0u) return __uint_as_float(hi);
    }
    return (float)x;
}
// The upper word of a double as an integer that orders like the double.
__device__ __forceinline__ int order_word(double x)
{
    const int h = __double2hiint(x);
    return h ^ ((h >> 31) & 0x7FFFFFFF);
}

// x' = x + dt v';  phi' = phi + dt Q(phi) w' with the 4x3 block of Sect. 2,
// renormalised (Sect. 3); periodic axes wrapped into [lo, hi).  With every
// conversion and comparison in FP64 (23 instructions a body) that bound the
// kernel: 4M bodies 180 us, now 110 (ncu, cold; their bytes take 96).
template <class R>
__global__ void k_integrate(int64_t n, double4_32a* __restrict__ pos_r, double4_32a* __restrict__ quat,
                            const R4<R>* __restrict__ vel, double dt, double3 lo, double3 L, int3 periodic,
                            DevInfo* info)
{
    bool bad = false;
    const int l0 = order_word(lo.x), h0 = order_word(lo.x + L.x), l1 = order_word(lo.y), h1 = order_word(lo.y + L.y),
              l2 = order_word(lo.z), h2 = order_word(lo.z + L.z);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        R4<R> v, w;
        ld_body(vel + 2 * i, v, w);
        double4_32a x = ld_d4(pos_r + i);
        x.x += dt * widen(v.x);
        x.y += dt * widen(v.y);
        x.z += dt * widen(v.z);
        double4_32a q = ld_d4(quat + i);
        {
            // quaternion update in the sweep precision (FP64 is scarce on this
            // GPU; orientations of spheres never feed back into the dynamics)
            using Q = R;
            Q qw = narrow_to<Q>(q.x), qx = narrow_to<Q>(q.y), qy = narrow_to<Q>(q.z), qz = narrow_to<Q>(q.w);
            const Q wx = w.x, wy = w.y, wz = w.z, hdt = (Q)(0.5 * dt);
            const Q dw = -qx * wx - qy * wy - qz * wz;
            const Q dx = qw * wx + qz * wy - qy * wz;
            const Q dy = -qz * wx + qw * wy + qx * wz;
            const Q dz = qy * wx - qx * wy + qw * wz;
            qw += hdt * dw;
            qx += hdt * dx;
            qy += hdt * dy;
            qz += hdt * dz;
            const Q inv = Q(1) / sqrt(qw * qw + qx * qx + qy * qy + qz * qz);
            q = make_double4_32a(widen(qw * inv), widen(qx * inv), widen(qy * inv), widen(qz * inv));
        }
        // periodic wrap into [lo, hi); only bodies that left the box pay for
        // fmod, and only those whose upper word does not show that they are inside for the test
        const int ox = order_word(x.x), oy = order_word(x.y), oz = order_word(x.z);
        if (periodic.x && !(ox > l0 && ox < h0) && !(x.x >= lo.x && x.x < lo.x + L.x)) {
            double s = fmod(x.x - lo.x, L.x);
            if (s < 0.0) s += L.x;
            x.x = lo.x + s;
        }
        if (periodic.y && !(oy > l1 && oy < h1) && !(x.y >= lo.y && x.y < lo.y + L.y)) {
            double s = fmod(x.y - lo.y, L.y);
            if (s < 0.0) s += L.y;
            x.y = lo.y + s;
        }
        if (periodic.z && !(oz > l2 && oz < h2) && !(x.z >= lo.z && x.z < lo.z + L.z)) {
            double s = fmod(x.z - lo.z, L.z);
            if (s < 0.0) s += L.z;
            x.z = lo.z + s;
        }
        // below 2^990 each, by the upper words, the sum is below 1e300
        const uint32_t big = max(max((uint32_t)__double2hiint(x.x) & 0x7FFFFFFFu, (uint32_t)__double2hiint(x.y) & 0x7FFFFFFFu),
                                 (uint32_t)__double2hiint(x.z) & 0x7FFFFFFFu);
        if (big >= 0x7DD00000u && !(fabs(x.x) + fabs(x.y) + fabs(x.z) <= 1e300)) bad = true;
        st_d4(pos_r + i, x);
        st_d4(quat + i, q);
    }
    if (bad) atomicOr(&info->err, kErrNaN);
}

nbgs_status run_integrate(nbgs_scene* s)
{
    if (s->composite) return run_integrate_comp(s);
    if (s->n == 0) return NBGS_OK;
    cudaStream_t st = s->stream;
    if (s->timing) cudaEventRecord(s->ev[6], st);
    const double3 lo = make_double3(s->prm.box_lo[0], s->prm.box_lo[1], s->prm.box_lo[2]);
    const double3 L = make_double3(s->prm.box_hi[0] - s->prm.box_lo[0], s->prm.box_hi[1] - s->prm.box_lo[1],
                                   s->prm.box_hi[2] - s->prm.box_lo[2]);
    const int3 per = make_int3(s->prm.periodic[0], s->prm.periodic[1], s->prm.periodic[2]);
    const int T = 256, gb = grid_for(s->n, T, 8, s->num_sms);
    if (s->fp32)
        k_integrate<float><<<gb, T, 0, st>>>(s->n, s->pos_r, s->quat, (const float4*)s->vel, s->prm.dt, lo, L, per,
                                             s->info);
    else
        k_integrate<double><<<gb, T, 0, st>>>(s->n, s->pos_r, s->quat, (const double4_32a*)s->vel, s->prm.dt, lo, L, per,
                                              s->info);
    if (s->timing) {
        s->phase_launches[3] += 1;
        cudaEventRecord(s->ev[7], st);
    }
    s->detected = s->coloured = false;
    return cuda_check(s, cudaGetLastError(), "integrate");
}

// ---------------------------------------------------------------------------
// state transfer: arrays on this GPU are read and written where they are;
// others go through the staging buffer, pos (3n) | quat (4n) | vel (3n) |
// angvel (3n).  4M bodies: the four copies beside each kernel took 125 us.
// ---------------------------------------------------------------------------
// Is [p, p + bytes) doubles in one allocation of this GPU?  (A copy of an array
// that ends before that fails; so it is left to the copy to say so.)
static bool on_device(const void* p, size_t bytes)
{
    if (((uintptr_t)p & 7u) != 0) return false;
    cudaPointerAttributes at;
    int dev = -1;
    if (cudaPointerGetAttributes(&at, p) != cudaSuccess || cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return false;
    }
    if (at.type != cudaMemoryTypeDevice || at.device != dev) return false;
    using Range = int (*)(unsigned long long*, size_t*, unsigned long long);
    static const Range range = [] {
        void* f = nullptr;
        cudaDriverEntryPointQueryResult q = cudaDriverEntryPointSymbolNotFound;
        if (cudaGetDriverEntryPointByVersion("cuMemGetAddressRange", &f, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess) {
            cudaGetLastError();
            f = nullptr;
        }
        return (Range)f;
    }();
    unsigned long long base = 0;
    size_t size = 0;
    if (!range || range(&base, &size, (unsigned long long)(uintptr_t)p) != 0) return false;
    return (unsigned long long)(uintptr_t)p + bytes <= base + size;
}

// Null arrays are left alone.
template <class R>
__global__ void k_unpack_state(int64_t n, const double* __restrict__ P, const double* __restrict__ Q,
                               const double* __restrict__ V, const double* __restrict__ W,
                               double4_32a* __restrict__ pos_r, double4_32a* __restrict__ quat,
                               R4<R>* __restrict__ vel)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        if (P) {
            double4_32a x = pos_r[i];
            x.x = P[3 * i];
            x.y = P[3 * i + 1];
            x.z = P[3 * i + 2];
            pos_r[i] = x;
        }
        if (Q) quat[i] = make_double4_32a(Q[4 * i], Q[4 * i + 1], Q[4 * i + 2], Q[4 * i + 3]);
        if (V) {
            R4<R> v = vel[2 * i];
            v.x = (R)V[3 * i];
            v.y = (R)V[3 * i + 1];
            v.z = (R)V[3 * i + 2];
            vel[2 * i] = v;
        }
        if (W) {
            R4<R> w = vel[2 * i + 1];
            w.x = (R)W[3 * i];
            w.y = (R)W[3 * i + 1];
            w.z = (R)W[3 * i + 2];
            vel[2 * i + 1] = w;
        }
    }
}

template <class R>
__global__ void k_pack_state(int64_t n, double* P, double* Q, double* V, double* W,
                             const double4_32a* __restrict__ pos_r, const double4_32a* __restrict__ quat,
                             const R4<R>* __restrict__ vel)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        if (P) {
            const double4_32a x = pos_r[i];
            P[3 * i] = x.x;
            P[3 * i + 1] = x.y;
            P[3 * i + 2] = x.z;
        }
        if (Q) {
            const double4_32a q = quat[i];
            Q[4 * i] = q.x;
            Q[4 * i + 1] = q.y;
            Q[4 * i + 2] = q.z;
            Q[4 * i + 3] = q.w;
        }
        if (V) {
            const R4<R> v = vel[2 * i];
            V[3 * i] = v.x;
            V[3 * i + 1] = v.y;
            V[3 * i + 2] = v.z;
        }
        if (W) {
            const R4<R> w = vel[2 * i + 1];
            W[3 * i] = w.x;
            W[3 * i + 1] = w.y;
            W[3 * i + 2] = w.z;
        }
    }
}

// Sect. 2: m = rho 4/3 pi r^3, I = 2/5 m r^2 (init), or explicit 1/m, 1/I.
template <class R>
__global__ void k_set_mass(int64_t n, const double* __restrict__ a, const double* __restrict__ b, int mode,
                           int has_a, int has_b, double4_32a* __restrict__ pos_r, R4<R>* __restrict__ vel,
                           uint8_t* __restrict__ finite, double* __restrict__ rmax_out)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        R4<R> v = vel[2 * i], w = vel[2 * i + 1];
        double im = v.w, iI = w.w;
        if (mode == 0) {  // a = radius, b = density
            const double r = a[i], rho = b[i];
            const double mass = rho * (4.0 / 3.0) * 3.14159265358979323846 * r * r * r;
            const double inertia = 0.4 * mass * r * r;
            im = mass > 0.0 ? 1.0 / mass : 0.0;
            iI = inertia > 0.0 ? 1.0 / inertia : 0.0;
            double4_32a x = pos_r[i];
            x.w = r;
            pos_r[i] = x;
        } else {
            if (has_a) im = a[i];
            if (has_b) iI = b[i];
        }
        v.w = (R)im;
        w.w = (R)iI;
        vel[2 * i] = v;
        vel[2 * i + 1] = w;
        finite[i] = (im > 0.0 || iI > 0.0) ? 1 : 0;
    }
}

template <class R>
static nbgs_status set_bodies_impl(nbgs_scene* s, const double* pos, const double* quat, const double* vel,
                                   const double* angvel)
{
    const int64_t n = s->n;
    cudaStream_t st = s->stream;
    const double* src[4] = {pos, quat, vel, angvel};
    const int64_t at[4] = {0, 3 * n, 7 * n, 10 * n}, len[4] = {3 * n, 4 * n, 3 * n, 3 * n};
    const char* what[4] = {"set pos", "set quat", "set vel", "set angvel"};
    for (int k = 0; k < 4; ++k) {
        if (!src[k] || on_device(src[k], len[k] * sizeof(double))) continue;
        nbgs_status rc = cuda_check(s, cudaMemcpyAsync(s->stage + at[k], src[k], len[k] * sizeof(double),
                                                       cudaMemcpyDefault, st), what[k]);
        if (rc != NBGS_OK) return rc;
        src[k] = s->stage + at[k];
    }
    const int T = 256;
    k_unpack_state<R><<<grid_for(n, T, 8, s->num_sms), T, 0, st>>>(n, src[0], src[1], src[2], src[3], s->pos_r,
                                                                   s->quat, (R4<R>*)s->vel);
    s->detected = s->coloured = false;
    return cuda_check(s, cudaGetLastError(), "set_bodies");
}

nbgs_status run_set_bodies(nbgs_scene* s, const double* pos, const double* quat, const double* vel,
                           const double* angvel)
{
    if (s->composite) return run_comp_set_bodies(s, pos, quat, vel, angvel);
    if (s->n == 0) return NBGS_OK;
    return s->fp32 ? set_bodies_impl<float>(s, pos, quat, vel, angvel) : set_bodies_impl<double>(s, pos, quat, vel, angvel);
}

nbgs_status run_get_bodies(nbgs_scene* s, double* pos, double* quat, double* vel, double* angvel)
{
    if (s->composite) return run_comp_get_bodies(s, pos, quat, vel, angvel);
    const int64_t n = s->n;
    if (n == 0) return NBGS_OK;
    cudaStream_t st = s->stream;
    double* const out[4] = {pos, quat, vel, angvel};
    const int64_t at[4] = {0, 3 * n, 7 * n, 10 * n}, len[4] = {3 * n, 4 * n, 3 * n, 3 * n};
    const char* what[4] = {"get pos", "get quat", "get vel", "get angvel"};
    double* dst[4];
    for (int k = 0; k < 4; ++k) {
        // arrays that overlap are written one after the other, by the copies
        bool alone = true;
        for (int q = 0; q < 4; ++q)
            alone = alone && (q == k || !out[q] || !out[k] || (uintptr_t)(out[q] + len[q]) <= (uintptr_t)out[k] ||
                              (uintptr_t)(out[k] + len[k]) <= (uintptr_t)out[q]);
        dst[k] = !out[k] ? nullptr : alone && on_device(out[k], len[k] * sizeof(double)) ? out[k] : s->stage + at[k];
    }
    const int T = 256;
    if (s->fp32)
        k_pack_state<float><<<grid_for(n, T, 8, s->num_sms), T, 0, st>>>(n, dst[0], dst[1], dst[2], dst[3], s->pos_r,
                                                                         s->quat, (const float4*)s->vel);
    else
        k_pack_state<double><<<grid_for(n, T, 8, s->num_sms), T, 0, st>>>(n, dst[0], dst[1], dst[2], dst[3], s->pos_r,
                                                                          s->quat, (const double4_32a*)s->vel);
    nbgs_status rc = cuda_check(s, cudaGetLastError(), "get_bodies");
    for (int k = 0; k < 4 && rc == NBGS_OK; ++k)
        if (out[k] && dst[k] != out[k])
            rc = cuda_check(s, cudaMemcpyAsync(out[k], dst[k], len[k] * sizeof(double), cudaMemcpyDefault, st), what[k]);
    if (rc == NBGS_OK) rc = cuda_check(s, cudaStreamSynchronize(st), "get_bodies");
    return rc;
}

nbgs_status run_set_mass(nbgs_scene* s, const double* a, const double* b, bool init, const double* radius,
                         const double* density)
{
    const int64_t n = s->n;
    if (n == 0) return NBGS_OK;
    cudaStream_t st = s->stream;
    double* A = s->stage;
    double* B = s->stage + n;
    const double* srcA = init ? radius : a;
    const double* srcB = init ? density : b;
    nbgs_status rc = NBGS_OK;
    if (srcA) rc = cuda_check(s, cudaMemcpyAsync(A, srcA, n * sizeof(double), cudaMemcpyDefault, st), "mass a");
    if (rc == NBGS_OK && srcB)
        rc = cuda_check(s, cudaMemcpyAsync(B, srcB, n * sizeof(double), cudaMemcpyDefault, st), "mass b");
    if (rc != NBGS_OK) return rc;
    const int T = 256;
    if (s->fp32)
        k_set_mass<float><<<grid_for(n, T, 8, s->num_sms), T, 0, st>>>(n, A, B, init ? 0 : 1, srcA != nullptr,
                                                                       srcB != nullptr, s->pos_r, (float4*)s->vel,
                                                                       s->finite, nullptr);
    else
        k_set_mass<double><<<grid_for(n, T, 8, s->num_sms), T, 0, st>>>(n, A, B, init ? 0 : 1, srcA != nullptr,
                                                                        srcB != nullptr, s->pos_r, (double4_32a*)s->vel,
                                                                        s->finite, nullptr);
    s->detected = s->coloured = false;
    return cuda_check(s, cudaGetLastError(), "set_mass_properties");
}

// ---------------------------------------------------------------------------
// contacts out: staging of 10 doubles per contact
// ---------------------------------------------------------------------------
__global__ void k_pack_contacts(int64_t m, const uint32_t* __restrict__ cstate, const double4_32a* __restrict__ cgeo,
                                const double4_32a* __restrict__ cimp, int solved, int32_t* __restrict__ col,
                                double* __restrict__ nrm, double* __restrict__ xi, double* __restrict__ imp)
{
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < m; c += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t sc = cstate[c];
        col[c] = sc == kUncoloured ? -1 : (int32_t)(sc & 0xFFu);
        const double4_32a g = cgeo[c];
        nrm[3 * c] = g.x;
        nrm[3 * c + 1] = g.y;
        nrm[3 * c + 2] = g.z;
        xi[c] = g.w;
        const double4_32a p = solved ? cimp[c] : make_double4_32a(0, 0, 0, 0);
        imp[3 * c] = p.x;
        imp[3 * c + 1] = p.y;
        imp[3 * c + 2] = p.z;
    }
}

nbgs_status run_get_contacts(nbgs_scene* s, int64_t cap, uint32_t* j1, uint32_t* j2, int32_t* colour, double* normal,
                             double* xi, double* impulse)
{
    const int64_t m = s->n_contacts < cap ? s->n_contacts : cap;
    if (m <= 0) return NBGS_OK;
    cudaStream_t st = s->stream;
    // 8 doubles per contact: colour (as int32 in a double slot), normal 3, xi, impulse 3
    double* buf = (double*)dev_alloc(s, (size_t)m * 8 * sizeof(double));
    if (!buf) return fail(s, NBGS_ENOMEM, "get_contacts: staging allocation failed");
    int32_t* col = (int32_t*)buf;
    double* nrm = buf + m;
    double* xiv = buf + 4 * m;
    double* imp = buf + 5 * m;
    if (!s->coloured && !s->solved) cudaMemsetAsync(s->cstate, 0xFF, m * sizeof(uint32_t), st);
    const int T = 256;
    k_pack_contacts<<<grid_for(m, T, 8, s->num_sms), T, 0, st>>>(m, s->cstate, s->cgeo, s->cimp, s->solved ? 1 : 0, col,
                                                                 nrm, xiv, imp);
    nbgs_status rc = cuda_check(s, cudaGetLastError(), "get_contacts");
    if (rc == NBGS_OK && j1) rc = cuda_check(s, cudaMemcpyAsync(j1, s->cj1, m * 4, cudaMemcpyDefault, st), "j1");
    if (rc == NBGS_OK && j2) rc = cuda_check(s, cudaMemcpyAsync(j2, s->cj2, m * 4, cudaMemcpyDefault, st), "j2");
    if (rc == NBGS_OK && colour) rc = cuda_check(s, cudaMemcpyAsync(colour, col, m * 4, cudaMemcpyDefault, st), "col");
    if (rc == NBGS_OK && normal)
        rc = cuda_check(s, cudaMemcpyAsync(normal, nrm, m * 24, cudaMemcpyDefault, st), "normal");
    if (rc == NBGS_OK && xi) rc = cuda_check(s, cudaMemcpyAsync(xi, xiv, m * 8, cudaMemcpyDefault, st), "xi");
    if (rc == NBGS_OK && impulse)
        rc = cuda_check(s, cudaMemcpyAsync(impulse, imp, m * 24, cudaMemcpyDefault, st), "impulse");
    if (rc == NBGS_OK) rc = cuda_check(s, cudaStreamSynchronize(st), "get_contacts");
    dev_free(s, buf);
    return rc;
}

}  // namespace nbgs
