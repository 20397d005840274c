// detect.cu -- contact detection (Sect. 4) on a uniform cell grid.
//
// Per step:
//   k_hull          h_i = dt(|v_i| + |w_i| r_i) + tau       eq. (expansionradius)
//                   + max h, max |v| (for the cell size and v_ref)
//   k_cell_keys     cell width >= 2 (r_max + h_max), dims per axis; every
//                   body's linear cell index and its rank in the cell
//   scan            first slot of every cell, from the cell counts
//   k_cell_scatter  bodies and their FP32 positions in cell order
//   k_narrow        per body: bodies in its own and the 13 cells ahead whose
//                   hulls intersect; wall hull tests
//   scan            contacts per body -> CSR offsets by j1
//   k_write_ends    canonical contacts, partners in ascending order
//   k_contact_geometry  their normals, gaps and lever lengths, for
//                   sphere-sphere and sphere-wall pairs, eq. (contactpos)
#include <algorithm>
#include <cmath>
#include <utility>

#include "nbgs_internal.cuh"

namespace nbgs {

int grid_for(int64_t work, int threads, int max_blocks_per_sm, int num_sms)
{
    int64_t b = (work + threads - 1) / threads;
    int64_t cap = (int64_t)max_blocks_per_sm * (num_sms > 0 ? num_sms : 1);
    if (b > cap) b = cap;
    if (b < 1) b = 1;
    return (int)b;
}

// ---------------------------------------------------------------------------
// exclusive scan of u32 (reduce -> scan block sums -> downsweep)
// ---------------------------------------------------------------------------
constexpr int kScanThreads = 256;
constexpr int kScanItems = 16;
constexpr int kScanTile = kScanThreads * kScanItems;

__device__ __forceinline__ uint32_t warp_incl_scan(uint32_t v)
{
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        uint32_t y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
    }
    return v;
}

// Exclusive block scan of one value per thread; returns the block total.
__device__ __forceinline__ uint32_t block_excl_scan(uint32_t v, uint32_t& excl)
{
    __shared__ uint32_t warp_tot[32];
    __shared__ uint32_t block_tot;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int nw = (blockDim.x + 31) >> 5;
    uint32_t inc = warp_incl_scan(v);
    if (lane == 31) warp_tot[wid] = inc;
    __syncthreads();
    if (wid == 0) {
        uint32_t t = lane < nw ? warp_tot[lane] : 0;
        uint32_t ti = warp_incl_scan(t);
        if (lane < nw) warp_tot[lane] = ti - t;
        if (lane == nw - 1) block_tot = ti;
    }
    __syncthreads();
    excl = warp_tot[wid] + inc - v;
    uint32_t total = block_tot;
    __syncthreads();
    return total;
}

// What a scan adds up: an array, or a body's contacts from its pair count and
// kept-wall mask.
struct ScanArray {
    const uint32_t* in;
    __device__ __forceinline__ uint32_t operator[](int64_t i) const { return in[i]; }
};
struct ScanRows {
    const uint32_t *pairs, *walls;
    __device__ __forceinline__ uint32_t operator[](int64_t i) const
    {
        return min(pairs[i], (uint32_t)kCandCap) + (uint32_t)__popc(walls[i]);
    }
};

template <class In>
__global__ void k_scan_reduce(In in, DCount nc, uint32_t* __restrict__ sums)
{
    const int64_t n = nc.get();
    const int64_t base = (int64_t)blockIdx.x * kScanTile;
    uint32_t acc = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        int64_t i = base + (int64_t)k * kScanThreads + threadIdx.x;
        if (i < n) acc += in[i];
    }
    uint32_t excl;
    uint32_t tot = block_excl_scan(acc, excl);
    if (threadIdx.x == 0) sums[blockIdx.x] = tot;
}

__global__ void k_scan_top(uint32_t* sums, int64_t nb)
{
    // single block: exclusive scan of the block sums in chunks
    uint32_t carry = 0;
    for (int64_t base = 0; base < nb; base += blockDim.x) {
        int64_t i = base + threadIdx.x;
        uint32_t v = i < nb ? sums[i] : 0;
        uint32_t excl;
        uint32_t tot = block_excl_scan(v, excl);
        if (i < nb) sums[i] = carry + excl;
        carry += tot;
    }
}

// top: the block sums have been scanned (k_scan_top); otherwise each block
// adds up the sums before its own, which for up to kScanSelf blocks costs
// less than a launch of its own.
constexpr int kScanSelf = 2048;

template <bool top, class In>
__global__ void k_scan_down(In in, uint32_t* out, DCount nc,
                            const uint32_t* __restrict__ sums, uint32_t* __restrict__ total_dst)
{
    __shared__ uint32_t tile[kScanTile];
    const int64_t n = nc.get();   // tiles past n hold zeros: the last block's total is the total
    const int64_t base = (int64_t)blockIdx.x * kScanTile;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        int64_t i = base + (int64_t)k * kScanThreads + threadIdx.x;
        tile[k * kScanThreads + threadIdx.x] = i < n ? in[i] : 0;
    }
    uint32_t before = 0;
    if (top) {
        before = sums[blockIdx.x];
    } else {
        uint32_t part = 0, excl;
        for (uint32_t i = threadIdx.x; i < blockIdx.x; i += kScanThreads) part += sums[i];
        before = block_excl_scan(part, excl);
    }
    __syncthreads();
    uint32_t loc[kScanItems];
    uint32_t acc = 0;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        loc[k] = acc;
        acc += tile[threadIdx.x * kScanItems + k];
    }
    uint32_t excl;
    uint32_t tot = block_excl_scan(acc, excl);
    const uint32_t off = before + excl;
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) tile[threadIdx.x * kScanItems + k] = loc[k] + off;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < kScanItems; ++k) {
        int64_t i = base + (int64_t)k * kScanThreads + threadIdx.x;
        if (i < n) out[i] = tile[k * kScanThreads + threadIdx.x];
    }
    if (blockIdx.x == gridDim.x - 1 && threadIdx.x == 0) {
        uint32_t total = before + tot;
        out[n] = total;
        if (total_dst) *total_dst = total;
    }
}

// out must hold n + 1 entries; out[n] receives the total (also *total_dst).
// A device-read count: the launch covers n.v entries (the capacity).
template <class In>
static nbgs_status exclusive_scan(nbgs_scene* s, In in, uint32_t* out, DCount n, uint32_t* total_dst)
{
    int64_t nb = (n.v + kScanTile - 1) / kScanTile;
    if (nb < 1) nb = 1;
    if (nb > s->scan_tmp_len) return fail(s, NBGS_EINVAL, "scan: block-sum buffer too small");
    k_scan_reduce<<<(unsigned)nb, kScanThreads, 0, s->stream>>>(in, n, s->scan_tmp);
    if (nb > kScanSelf) {
        k_scan_top<<<1, 1024, 0, s->stream>>>(s->scan_tmp, nb);
        k_scan_down<true, In><<<(unsigned)nb, kScanThreads, 0, s->stream>>>(in, out, n, s->scan_tmp, total_dst);
    } else {
        k_scan_down<false, In><<<(unsigned)nb, kScanThreads, 0, s->stream>>>(in, out, n, s->scan_tmp, total_dst);
    }
    return cuda_check(s, cudaGetLastError(), "scan");
}

nbgs_status exclusive_scan_u32(nbgs_scene* s, const uint32_t* in, uint32_t* out, DCount n, uint32_t* total_dst)
{
    return exclusive_scan(s, ScanArray{in}, out, n, total_dst);
}

nbgs_status exclusive_scan_u32(nbgs_scene* s, const uint32_t* in, uint32_t* out, int64_t n, uint32_t* total_dst)
{
    return exclusive_scan_u32(s, in, out, DCount{n, nullptr}, total_dst);
}

// ---------------------------------------------------------------------------
// detection kernels
// ---------------------------------------------------------------------------
struct GridArgs {
    double lo[3], hi[3];
    int periodic[3];
    int dims_max[3];
    double r_max, dt, tau;
    float Lf[3];         // box extents in FP32
    float margin;        // FP32 pre-filter margin: 1e-4 + 1e-6 max(L)
    double pos_err;      // bound on the error of an FP32 relative position (2^-22 max(L))
    // FP32 wall pre-filter: plane k as n . (x - lo) + pc[k] (= n . x - c),
    // margin 1e-4 + 4e-6 (max(L) + max |pc|)
    float pn[kMaxPlanes][3];
    float pc[kMaxPlanes];
    float tauf, wmargin;
    // FP32 cone pre-filter: apex relative to lo, axis, sin, cos, s_o, s_t;
    // margin 1e-4 + 1e-5 (max(L) + max |apex - lo|)
    float ca_apex[kMaxCones][3], ca_axis[kMaxCones][3], ca_sc[kMaxCones][4];
    float cmargin;
};

__device__ __forceinline__ double norm_exact(double x, double y, double z)
{
    return xsqrt(xadd(xadd(xmul(x, x), xmul(y, y)), xmul(z, z)));
}

// a / b rounded to nearest, given y = 1/b rounded to nearest: the quotient
// q = RN(a y) is within one ulp of a / b, the remainder a - b q is exact in
// one fused multiply-add, and RN(q + (a - b q) y) is the correctly rounded
// quotient (Markstein's theorem, IBM J. Res. Dev. 34(1), 1990; Muller et
// al., Handbook of Floating-Point Arithmetic, the chapter on division with
// an FMA).  The theorem excludes underflow: tiny numerators take the division
// itself, as does the caller for a tiny or huge b; a zero (every pair inside a
// lattice plane has one) is its own quotient, b being positive, and does not
// take its warp through the division (three of them made 93 FP64 instructions
// of a dense lattice's 45 a pair).
__device__ __forceinline__ double div_by(double a, double b, double y)
{
    const uint32_t e = (uint32_t)__double2hiint(a) & 0x7FFFFFFFu;
    const bool zero = (e | (uint32_t)__double2loint(a)) == 0u;
    if (e < 0x07B00000u && !zero) return xdiv(a, b);   // |a| < 2^-900
    const double q = __dmul_rn(a, y);
    const double r = __fma_rn(-q, b, a);
    const double v = __fma_rn(r, y, q);
    return zero ? a : v;   // keeps its sign
}

// Sphere pair geometry of eq. (contactpos) from the centre difference
// (dx, dy, dz) = x_i - x_j: d = |x_i - x_j| and the unit normal
// n = (x_i - x_j) / d, every operation rounded to nearest as written (the
// three quotients share one correctly rounded reciprocal of d); coincident
// centres take n = (0, 0, 1).
__device__ __forceinline__ double pair_normal(double dx, double dy, double dz, double n[3])
{
    const double d = norm_exact(dx, dy, dz);
    // 2^-1000 <= d < 2^1000, by its upper word (d is not negative)
    if ((uint32_t)__double2hiint(d) - 0x01700000u < 0x7D000000u) {
        const double y = __drcp_rn(d);
        n[0] = div_by(dx, d, y);
        n[1] = div_by(dy, d, y);
        n[2] = div_by(dz, d, y);
    } else if (d > 0.0) {
        n[0] = xdiv(dx, d);
        n[1] = xdiv(dy, d);
        n[2] = xdiv(dz, d);
    } else {
        n[0] = 0.0;
        n[1] = 0.0;
        n[2] = 1.0;
    }
    return d;
}

// Composite particles: the members' world positions X + R(q) d (FP64, each
// operation rounded as written: the contact geometry depends on them bit for
// bit), their bodies' hulls h = dt (|v| + |w| r_bound) + tau (eq.
// expansionradius with the bounding radius) and the FP32 copies for the cell
// grid, wrapped into the box on periodic axes (the FP64 positions stay
// unwrapped; the exact tests take minimum images of differences).
template <class R>
__global__ void k_member_update(int64_t n, const uint32_t* __restrict__ mbody, const double4_32a* __restrict__ moff,
                                const double4_32a* __restrict__ bpos, const double4_32a* __restrict__ bquat,
                                const R4<R>* __restrict__ bvel, double dt, double tau,
                                double4_32a* __restrict__ pos_r, double* __restrict__ hull, float4* __restrict__ p32,
                                GridArgs g, DevInfo* info)
{
    double hmax = 0.0, vmax = 0.0;
    bool bad = false;
    for (int64_t m = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; m < n; m += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t b = mbody[m];
        const double4_32a X = ld_d4(bpos + b), q = ld_d4(bquat + b), d = ld_d4(moff + m);
        const R4<R> v = bvel[4 * (int64_t)b], w = bvel[4 * (int64_t)b + 1];
        // R(q) rows, as 1 - 2 (y^2 + z^2), 2 (xy - wz), ... (unit quaternion)
        const double qw = q.x, qx = q.y, qy = q.z, qz = q.w;
        const double r00 = xsub(1.0, xmul(2.0, xadd(xmul(qy, qy), xmul(qz, qz))));
        const double r01 = xmul(2.0, xsub(xmul(qx, qy), xmul(qw, qz)));
        const double r02 = xmul(2.0, xadd(xmul(qx, qz), xmul(qw, qy)));
        const double r10 = xmul(2.0, xadd(xmul(qx, qy), xmul(qw, qz)));
        const double r11 = xsub(1.0, xmul(2.0, xadd(xmul(qx, qx), xmul(qz, qz))));
        const double r12 = xmul(2.0, xsub(xmul(qy, qz), xmul(qw, qx)));
        const double r20 = xmul(2.0, xsub(xmul(qx, qz), xmul(qw, qy)));
        const double r21 = xmul(2.0, xadd(xmul(qy, qz), xmul(qw, qx)));
        const double r22 = xsub(1.0, xmul(2.0, xadd(xmul(qx, qx), xmul(qy, qy))));
        double4_32a p;
        p.x = xadd(X.x, xadd(xadd(xmul(r00, d.x), xmul(r01, d.y)), xmul(r02, d.z)));
        p.y = xadd(X.y, xadd(xadd(xmul(r10, d.x), xmul(r11, d.y)), xmul(r12, d.z)));
        p.z = xadd(X.z, xadd(xadd(xmul(r20, d.x), xmul(r21, d.y)), xmul(r22, d.z)));
        p.w = d.w;
        st_d4(pos_r + m, p);
        const double nv = norm_exact((double)v.x, (double)v.y, (double)v.z);
        const double nw = norm_exact((double)w.x, (double)w.y, (double)w.z);
        const double h = xadd(xmul(dt, xadd(nv, xmul(nw, X.w))), tau);
        hull[m] = h;
        double rel[3] = {p.x - g.lo[0], p.y - g.lo[1], p.z - g.lo[2]};
        for (int a = 0; a < 3; ++a) {
            const double L = g.hi[a] - g.lo[a];
            if (g.periodic[a] && !(rel[a] >= 0.0 && rel[a] < L)) {
                double sft = fmod(rel[a], L);
                if (sft < 0.0) sft += L;
                rel[a] = sft;
            }
        }
        p32[m] = make_float4((float)rel[0], (float)rel[1], (float)rel[2], (float)(p.w + h));
        if (!(h <= 1e300)) bad = true;
        hmax = fmax(hmax, h);
        vmax = fmax(vmax, nv);
    }
    __shared__ double sh[2][32];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int o = 16; o > 0; o >>= 1) {
        hmax = fmax(hmax, __shfl_down_sync(0xffffffffu, hmax, o));
        vmax = fmax(vmax, __shfl_down_sync(0xffffffffu, vmax, o));
    }
    if (lane == 0) {
        sh[0][wid] = hmax;
        sh[1][wid] = vmax;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < (int)(blockDim.x >> 5); ++k) {
            hmax = fmax(hmax, sh[0][k]);
            vmax = fmax(vmax, sh[1][k]);
        }
        atomicMax(&info->hmax_bits, (unsigned long long)__double_as_longlong(hmax));
        atomicMax(&info->vmax_bits, (unsigned long long)__double_as_longlong(vmax));
    }
    if (bad) atomicOr(&info->err, kErrNaN);
}

// Hull radius of eq. (expansionradius), h = dt (|v| + |w| r) + tau, rounded
// as the FP64 step computes it: for a sphere from its velocities, where a
// decision needs it (only those contacts pay for its two square roots), for a
// composite member from the member hulls.
struct HullView {
    const double* hull;   // member hulls (composites), else null
    const void* vel;      // (v, 1/m), (w, 1/I) per sphere
    int fp32;             // in FP32 or FP64
    double dt, tau;
};

template <class R>
__device__ __forceinline__ double norm2_exact(const R4<R>& v)
{
    const double x = v.x, y = v.y, z = v.z;
    return xadd(xadd(xmul(x, x), xmul(y, y)), xmul(z, z));
}

template <bool Together>   // a copy for either narrow phase: ptxas 13.0 fails on two kernels calling one
__device__ __noinline__ double hull_of(const HullView& H, uint32_t x, double r)
{
    if (H.hull) return H.hull[x];
    double v2, w2;
    if (H.fp32) {
        float4 v, w;
        ld_body((const float4*)H.vel + 2 * (int64_t)x, v, w);
        v2 = norm2_exact<float>(v);
        w2 = norm2_exact<float>(w);
    } else {
        double4_32a v, w;
        ld_body((const double4_32a*)H.vel + 2 * (int64_t)x, v, w);
        v2 = norm2_exact<double>(v);
        w2 = norm2_exact<double>(w);
    }
    return xadd(xmul(H.dt, xadd(xsqrt(v2), xmul(xsqrt(w2), r))), H.tau);
}

// Per sphere: the FP32 position relative to the box corner and the reach r +
// h with h in FP32 (cell keys and the narrow phase's screens run on these; the
// FP32 hull is within 1e-6 of h relative, inside the screens' margins), and an
// upper bound of the largest hull for the grid.  v_ref wants max |v| exactly:
// the square root of the largest FP64 |v|^2, which only the bodies whose FP32
// |v|^2 (off by less than 4e-7 relative) is within 1e-6 of the block's largest
// can have; those few are looked at again.  FP64 arithmetic occupies this GPU's
// FP64 units for 16 cycles per warp and SM, so a square per body and component
// was most of this kernel's time: 4M bodies, 249 -> 66 us (ncu, cold).
template <class R>
__global__ void k_hull(int64_t n, const R4<R>* __restrict__ vel, const double4_32a* __restrict__ pos_r, double dt,
                       double tau, float4* __restrict__ p32, GridArgs g, DevInfo* info,
                       const uint32_t* __restrict__ scene_of, unsigned long long* __restrict__ scene_vmax)
{
    float hmax = 0.f, v2max = 0.f;
    bool bad = false;
    const float dtf = (float)dt, tauf = (float)tau;
    const int64_t first = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
    // by warps, so that the lanes with a body are known (the votes below)
    for (int64_t i0 = first - (threadIdx.x & 31); i0 < n; i0 += stride) {
        const int64_t i = i0 + (threadIdx.x & 31);
        if (i >= n) break;
        R4<R> v, w;
        ld_body(vel + 2 * i, v, w);
        const double4_32a x = ld_d4(pos_r + i);
        const float vx = (float)v.x, vy = (float)v.y, vz = (float)v.z, wx = (float)w.x, wy = (float)w.y, wz = (float)w.z;
        const float v2 = vx * vx + vy * vy + vz * vz, w2 = wx * wx + wy * wy + wz * wz;
        const float rf = (float)x.w, h32 = dtf * (sqrtf(v2) + sqrtf(w2) * rf) + tauf;
        p32[i] = make_float4((float)(x.x - g.lo[0]), (float)(x.y - g.lo[1]), (float)(x.z - g.lo[2]), rf + h32);
        // beyond FP32: NaN, Inf, or squares too large for it
        if (!(v2 <= 1e38f && w2 <= 1e38f) && !(norm2_exact<R>(v) <= 1e300 && norm2_exact<R>(w) <= 1e300)) bad = true;
        if (scene_of) {   // per-scene max |v|^2 (v_ref); the filters only save FP64 squares and atomics
            const uint32_t sc = scene_of[i], act = n - i0 < 32 ? (1u << (int)(n - i0)) - 1u : 0xffffffffu;
            // a warp's bodies are mostly of one scene: only its fastest can count
            // (all of them asked for an atomic while the maxima were still low);
            // a NaN is nobody's maximum
            bool asks = true;
            if (__match_any_sync(act, sc) == act)
                asks = v2 >= __uint_as_float(__reduce_max_sync(act, v2 == v2 ? __float_as_uint(v2) : 0u)) * (1.f - 1e-6f) -
                                 1e-30f;
            unsigned long long* dst = scene_vmax + sc;
            if (asks &&
                !((float)__longlong_as_double((long long)*(volatile unsigned long long*)dst) > v2 * (1.f + 1e-6f) + 1e-30f)) {
                const unsigned long long bits = (unsigned long long)__double_as_longlong(norm2_exact<R>(v));
                if (bits > *(volatile unsigned long long*)dst) atomicMax(dst, bits);
            }
        }
        hmax = fmaxf(hmax, h32);
        v2max = fmaxf(v2max, v2);
    }
    __shared__ float sh[2][32];
    __shared__ float s_v2;
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = (int)(blockDim.x >> 5);
    const float own = v2max;
    for (int o = 16; o > 0; o >>= 1) {
        hmax = fmaxf(hmax, __shfl_xor_sync(0xffffffffu, hmax, o));
        v2max = fmaxf(v2max, __shfl_xor_sync(0xffffffffu, v2max, o));
    }
    if (lane == 0) {
        sh[0][wid] = hmax;
        sh[1][wid] = v2max;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < nw; ++k) {
            hmax = fmaxf(hmax, sh[0][k]);
            v2max = fmaxf(v2max, sh[1][k]);
        }
        s_v2 = v2max;
        // 1e-5 above the FP32 hulls is above the exact ones (non-negative doubles order like their bits)
        atomicMax(&info->hmax_bits, (unsigned long long)__double_as_longlong((double)hmax * (1.0 + 1e-5)));
    }
    __syncthreads();
    const float near = s_v2 > 1e-30f ? s_v2 * (1.f - 1e-6f) : 0.f;   // squares that underflow: look at all
    if (own >= near) {
        double best = 0.0;
        for (int64_t i = first; i < n; i += stride) {
            R4<R> v, w;
            ld_body(vel + 2 * i, v, w);
            const float vx = (float)v.x, vy = (float)v.y, vz = (float)v.z;
            if (vx * vx + vy * vy + vz * vz >= near) best = fmax(best, norm2_exact<R>(v));
        }
        atomicMax(&info->vmax_bits, (unsigned long long)__double_as_longlong(xsqrt(best)));
    }
    if (bad) atomicOr(&info->err, kErrNaN);
}

__device__ __forceinline__ int cell_coord(float x, float inv_w, int d)
{
    const float f = floorf(x * inv_w);
    return f < 0.f ? 0 : (f > (float)(d - 1) ? d - 1 : (int)f);
}

// The cell grid of the step (every block works it out, the first one notes it
// down), the cell of every body and its rank among the cell's bodies, in the
// order the counter served them: where in the cell's range of slots a body
// lands does not matter to anything that follows.
__global__ void k_cell_keys(int64_t n, const float4* __restrict__ p32, GridArgs g, DevInfo* info,
                            uint32_t* __restrict__ keys, uint32_t* __restrict__ rank, uint32_t* __restrict__ cnt)
{
    __shared__ int s_d[3];
    __shared__ float s_inv[3];
    if (threadIdx.x < 3) {
        const int a = threadIdx.x;
        const double hmax = __longlong_as_double((long long)info->hmax_bits);
        // any kept pair has d <= r_a + r_b + h_a + h_b <= 2 (r_max + h_max); the
        // cell keys come from FP32 positions with error <= pos_err, so a cell at
        // least need + 4 pos_err wide keeps every such pair in adjacent cells
        const double need = 2.0 * (g.r_max + hmax) * (1.0 + 1e-9) + 4.0 * g.pos_err + 1e-300;
        const double L = g.hi[a] - g.lo[a];
        const double dd = floor(L / need);
        const int d = dd < 1.0 ? 1 : (dd > (double)g.dims_max[a] ? g.dims_max[a] : (int)dd);
        s_d[a] = d;
        s_inv[a] = (float)(d / L);
        if (blockIdx.x == 0) {
            if (g.periodic[a] && d < 3) atomicOr(&info->err, kErrGrid);
            info->dims[a] = d;
            info->cell_w[a] = L / d;
            info->inv_wf[a] = s_inv[a];
        }
    }
    __syncthreads();
    const int d0 = s_d[0], d1 = s_d[1], d2 = s_d[2];
    const float i0 = s_inv[0], i1 = s_inv[1], i2 = s_inv[2];
    if (blockIdx.x == 0 && threadIdx.x == 0) info->ncells = (uint32_t)d0 * (uint32_t)d1 * (uint32_t)d2;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const float4 p = p32[i];
        const int cx = cell_coord(p.x, i0, d0), cy = cell_coord(p.y, i1, d1), cz = cell_coord(p.z, i2, d2);
        const uint32_t k = ((uint32_t)cz * (uint32_t)d1 + (uint32_t)cy) * (uint32_t)d0 + (uint32_t)cx;
        keys[i] = k;
        rank[i] = atomicAdd(&cnt[k], 1u);
    }
}

// Bodies and their FP32 positions in cell order, so that the narrow phase
// reads each cell's candidates contiguously.  A counting sort: against the
// radix sort of (cell, body) pairs of before, with its three or four passes
// of five kernels, 4M bodies take 30 + 60 us instead of 430 (ncu, cold).
__global__ void k_cell_scatter(int64_t n, const uint32_t* __restrict__ keys, const uint32_t* __restrict__ rank,
                               const uint32_t* __restrict__ cell_start, const float4* __restrict__ p32,
                               uint32_t* __restrict__ svals, float4* __restrict__ p32s)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t s = cell_start[keys[i]] + rank[i];
        svals[s] = (uint32_t)i;
        p32s[s] = p32[i];
    }
}

// Minimum-image difference a - b along one axis (periodic: |d| <= L/2).
__device__ __forceinline__ double min_image(double d, int periodic, double L)
{
    // |d| <= L / 2 is read off the upper words for all but the pairs across a
    // face: FP64 comparisons would cost as much as the arithmetic
    if (periodic && ((uint32_t)__double2hiint(d) & 0x7FFFFFFFu) >= (uint32_t)__double2hiint(L) - 0x00100000u) {
        const double half = xmul(0.5, L);
        if (d > half) d = xsub(d, L);
        else if (d < -half) d = xadd(d, L);
    }
    return d;
}

// Distance from x to cone C, worked in the half-plane through the axis and
// x: zeta = height above the apex along the axis, rho = distance from the
// axis, e = unit radial direction.  A generatrix runs along (sin a, cos a)
// in (rho, zeta); the face is its segment s in [s_o, s_t], the solid lies
// outside, and the face's inward unit normal is (-cos a, sin a).  The foot
// of x on the generatrix is at s = rho sin a + zeta cos a.  Face:
// sd = zeta sin a - rho cos a, n = sin a axis - cos a e.  Below the face
// (s < s_o) the orifice rim (rho_o, zeta_o) = s_o (sin a, cos a) is
// nearest: sd = |(rho - rho_o, zeta - zeta_o)|, n along that difference.
// On the axis (rho = 0) the normal is the axis.  Returns 0 above the
// frustum (no contact), 1 on the face, 2 at the rim.  Every operation is
// rounded to nearest, in this order, so that the contact sets are exact.
__device__ __forceinline__ int cone_distance(const Cone& C, const double4_32a& x, double& sd, double n[3])
{
    const double d0 = xsub(x.x, C.apex[0]), d1 = xsub(x.y, C.apex[1]), d2 = xsub(x.z, C.apex[2]);
    const double zeta = xadd(xadd(xmul(d0, C.axis[0]), xmul(d1, C.axis[1])), xmul(d2, C.axis[2]));
    double e0 = xsub(d0, xmul(zeta, C.axis[0])), e1 = xsub(d1, xmul(zeta, C.axis[1])),
           e2 = xsub(d2, xmul(zeta, C.axis[2]));
    const double rho = xsqrt(xadd(xadd(xmul(e0, e0), xmul(e1, e1)), xmul(e2, e2)));
    const double sg = xadd(xmul(rho, C.sa), xmul(zeta, C.ca));
    if (sg > C.s_t) return 0;
    if (rho > 0.0) {
        e0 = xdiv(e0, rho);
        e1 = xdiv(e1, rho);
        e2 = xdiv(e2, rho);
    }
    if (sg >= C.s_o) {
        sd = xsub(xmul(zeta, C.sa), xmul(rho, C.ca));
        if (rho > 0.0) {
            n[0] = xsub(xmul(C.sa, C.axis[0]), xmul(C.ca, e0));
            n[1] = xsub(xmul(C.sa, C.axis[1]), xmul(C.ca, e1));
            n[2] = xsub(xmul(C.sa, C.axis[2]), xmul(C.ca, e2));
        } else {
            n[0] = C.axis[0];
            n[1] = C.axis[1];
            n[2] = C.axis[2];
        }
        return 1;
    }
    const double drho = xsub(rho, xmul(C.s_o, C.sa)), dzeta = xsub(zeta, xmul(C.s_o, C.ca));
    const double dist = xsqrt(xadd(xmul(drho, drho), xmul(dzeta, dzeta)));
    sd = dist;
    if (dist > 0.0 && rho > 0.0) {
        n[0] = xdiv(xadd(xmul(drho, e0), xmul(dzeta, C.axis[0])), dist);
        n[1] = xdiv(xadd(xmul(drho, e1), xmul(dzeta, C.axis[1])), dist);
        n[2] = xdiv(xadd(xmul(drho, e2), xmul(dzeta, C.axis[2])), dist);
    } else {
        n[0] = C.axis[0];
        n[1] = C.axis[1];
        n[2] = C.axis[2];
    }
    return 2;
}

// The same distance in FP32 from the relative position q (the pre-filter;
// the distance is continuous across the face/rim boundary, so a case taken
// differently under rounding changes it little).  Returns a huge value
// above the frustum.
__device__ __forceinline__ float cone_distance_f(const GridArgs& g, int k, const float4& q)
{
    const float d0 = q.x - g.ca_apex[k][0], d1 = q.y - g.ca_apex[k][1], d2 = q.z - g.ca_apex[k][2];
    const float* ax = g.ca_axis[k];
    const float sa = g.ca_sc[k][0], ca = g.ca_sc[k][1], so = g.ca_sc[k][2], st = g.ca_sc[k][3];
    const float zeta = d0 * ax[0] + d1 * ax[1] + d2 * ax[2];
    const float e0 = d0 - zeta * ax[0], e1 = d1 - zeta * ax[1], e2 = d2 - zeta * ax[2];
    const float rho = sqrtf(e0 * e0 + e1 * e1 + e2 * e2);
    const float sg = rho * sa + zeta * ca;
    if (sg > st + g.cmargin) return 3.0e38f;
    if (sg >= so) return zeta * sa - rho * ca;
    const float dr = rho - so * sa, dz = zeta - so * ca;
    return sqrtf(dr * dr + dz * dz);
}

__device__ __forceinline__ bool wall_kept(const double nrm[3], double c, double4_32a p, double h, double tau, double& sd,
                                          double& xi)
{
    sd = xsub(xadd(xadd(xmul(nrm[0], p.x), xmul(nrm[1], p.y)), xmul(nrm[2], p.z)), c);
    xi = xsub(sd, p.w);
    return xi <= xadd(h, tau);
}

// Hull-intersecting pairs.  Every body (in cell order) looks at the bodies
// behind it in its own cell and at the 13 neighbour cells ahead (after it in
// z, y, x), so that each pair is tested once; the pair joins the list of its
// lower body through that body's counter, and k_write_ends puts each list
// into ascending order.  cs[c] is the first slot of cell c for every cell
// (cs[ncells] = n), so the cells x - 1 .. x + 1 of a (y, z) row are one
// contiguous range; a periodic image adds one constant shift to a whole
// range.  The kernel is bound by the instructions of the screens where pairs
// are few, and by the lists' atomics where they are many: with all 27 cells
// searched for both bodies of a pair, nested loops and the list in the
// thread, 4M gas bodies took 574 us and 1M packed ones 145 (ncu, cold), this
// way 368 and 213; the packed scene's solve takes 8 ms.  A late pile of 1M
// composites, 16.4M pairs: 1.74 ms before and 1.69 now (3.74 with each lane's
// queue worked off alone, see below).
//
// The search is a loop of FP32 screens over the rows' slots, run together
// (the lanes of a warp differ in the lengths of the rows by more than in
// their sum); the pairs that pass wait in a queue in shared memory, so that
// the lanes work them off together.  A lane whose queue is full works it off
// alone, which is rare among spheres; the members of packed composites, each of
// which meets its own body's too, fill theirs at different times and would wait
// for one another.  There (Together) the warp votes after every two screens and
// works all queues off when one is nearly full: detection of a pile of 1M
// composites, 5.6M contacts 2.68 -> 2.43 ms, 16.4M 5.70 -> 3.60; but 2.0M (0.65 a
// member) 1.55 -> 1.65, a gas of 16M spheres 2.66 -> 3.10, hence 3 contacts to 2
// members at the last detection as the line, and spheres never (1M in two sizes
// 0.88 -> 0.99, though 0.51 -> 0.47 in a pile).
constexpr int kNarrowThreads = 128, kNarrowRows = 5, kNarrowQueue = 8;
constexpr uint32_t kSurePair = 1u << 31;   // of a queued slot: kept without the FP64 test

// Sect. 4: is the pair kept?  Its lower and upper body; R is the sum of
// their FP32 reaches.
template <bool Together>
__device__ __noinline__ bool exact_pair(const HullView& H, const GridArgs& g, const double4_32a* __restrict__ pos_r,
                                        uint32_t lo, uint32_t hi, float R)
{
    const double4_32a pl = pos_r[lo], ph = pos_r[hi];
    const double dx3 = min_image(xsub(pl.x, ph.x), g.periodic[0], g.hi[0] - g.lo[0]);
    const double dy3 = min_image(xsub(pl.y, ph.y), g.periodic[1], g.hi[1] - g.lo[1]);
    const double dz3 = min_image(xsub(pl.z, ph.z), g.periodic[2], g.hi[2] - g.lo[2]);
    // The differences now hold no rounding of large coordinates: their FP32
    // square is within 4e-7 of d^2 and R within 1.2e-6 of the FP64 sum, which
    // leaves the FP64 square roots (d's, and the hulls' four) to the pairs
    // within 2e-6 of it.
    const float gx = (float)dx3, gy = (float)dy3, gz = (float)dz3;
    const float d2g = gx * gx + gy * gy + gz * gz, r2 = R * R;
    if (R > 1e-15f && R < 1e15f) {
        if (d2g > r2 * (1.f + 5e-6f)) return false;
        if (d2g < r2 * (1.f - 5e-6f)) return true;
    }
    const double d = norm_exact(dx3, dy3, dz3);
    return xsub(xsub(d, pl.w), ph.w) <= xadd(hull_of<Together>(H, lo, pl.w), hull_of<Together>(H, hi, ph.w));
}

// Neighbour index along one axis: the cell and the shift of the periodic
// image (the image of cell d - 1 left of cell 0 sits at -L); false when the
// cell lies outside a bounded axis.
__device__ __forceinline__ bool axis_cell(int c, int d, int periodic, float Lf, int& out, float& shift)
{
    shift = 0.f;
    if (c >= 0 && c < d) {
        out = c;
        return true;
    }
    if (!periodic || d < 3) return false;
    out = c < 0 ? c + d : c - d;
    shift = c < 0 ? Lf : -Lf;
    return true;
}

template <bool Together>
__global__ void __launch_bounds__(kNarrowThreads)
k_narrow(int64_t n, const uint32_t* __restrict__ svals, const double4_32a* __restrict__ pos_r,
         const __grid_constant__ HullView H, const float4* __restrict__ p32s, const uint32_t* __restrict__ cs,
         const __grid_constant__ GridArgs g, const __grid_constant__ Planes planes, SceneView V, DevInfo* info,
         uint32_t* __restrict__ cand, uint32_t* __restrict__ pair_cnt, uint32_t* __restrict__ wall_mask)
{
    __shared__ uint32_t s_t0[kNarrowRows][kNarrowThreads], s_t1[kNarrowRows][kNarrowThreads];
    __shared__ float2 s_yz[kNarrowRows][kNarrowThreads];   // y and z relative to the row's image
    __shared__ uint32_t s_q[kNarrowQueue][kNarrowThreads];
    const int tid = threadIdx.x;
    const int d0 = info->dims[0], d1 = info->dims[1], d2 = info->dims[2];
    const float i0 = info->inv_wf[0], i1 = info->inv_wf[1], i2 = info->inv_wf[2];
    const bool wrap_x = g.periodic[0] && d0 >= 3;
    const float margin =
        2.0 * (g.r_max + __longlong_as_double((long long)info->hmax_bits)) < 50.0 ? g.margin : 1e30f;
    // Together: by warps, whose lanes without a body only take part in the votes
    for (int64_t s0 = blockIdx.x * (int64_t)blockDim.x + (Together ? tid & ~31 : tid); s0 < n;
         s0 += (int64_t)gridDim.x * blockDim.x) {
        const bool live = !Together || s0 + (tid & 31) < n;
        const int64_t s = !Together ? s0 : live ? s0 + (tid & 31) : n - 1;
        const uint32_t i = svals[s];
        const uint32_t si = V.batch ? V.scene_of[i] : 0u;
        const float4 qi = p32s[s];
        // its cell, as k_cell_keys has it
        const int cx = cell_coord(qi.x, i0, d0), cy = cell_coord(qi.y, i1, d1), cz = cell_coord(qi.z, i2, d2);
        const int xlo = cx > 0 ? cx - 1 : 0, xhi = cx + 1 < d0 ? cx + 1 : d0 - 1;
        // the rows ahead: the rest of its own, (y + 1), and three in z + 1
#pragma unroll
        for (int k = 0; k < kNarrowRows; ++k) {
            int z, y;
            float sy = 0.f, sz = 0.f;
            uint32_t t0 = 0, t1 = 0;
            if (axis_cell(cz + (k > 1), d2, g.periodic[2], g.Lf[2], z, sz) &&
                axis_cell(cy + (k > 1 ? k - 3 : k), d1, g.periodic[1], g.Lf[1], y, sy)) {
                const uint32_t row = ((uint32_t)z * (uint32_t)d1 + (uint32_t)y) * (uint32_t)d0;
                t0 = k == 0 ? (uint32_t)s + 1u : cs[row + xlo];
                t1 = cs[row + xhi + 1];
            }
            s_yz[k][tid] = make_float2(qi.y + sy, qi.z + sz);
            s_t0[k][tid] = t0;
            s_t1[k][tid] = t1;
        }
        int nq = 0;
        auto work_off = [&]() {
            for (int m = 0; m < nq; ++m) {
                const uint32_t q = s_q[m][tid], t = q & ~kSurePair;
                const uint32_t j = svals[t];
                if (V.batch && V.scene_of[j] != si) continue;   // scenes never touch
                if (V.body_of && V.body_of[j] == V.body_of[i]) continue;   // nor members of one body
                const uint32_t lo = min(i, j), hi = max(i, j);
                if (!(q & kSurePair) && !exact_pair<Together>(H, g, pos_r, lo, hi, qi.w + p32s[t].w)) continue;
                const uint32_t slot = atomicAdd(&pair_cnt[lo], 1u);
                if (slot < (uint32_t)kCandCap) {
                    cand[(int64_t)lo * kCandCap + slot] = hi;
                } else {
                    atomicOr(&info->err, kErrCand);
                    atomicMax(&info->cand_need, slot + 1u);
                }
            }
            nq = 0;
        };
        // Conservative FP32 screens (FP64 throughput is scarce on this GPU).
        // R = r_a + h_a + r_b + h_b bounds d for every kept pair.  The FP32
        // relative positions are off by at most pos_err per coordinate, the
        // periodic shift adds an ulp of L, so the FP32 distance is within
        // 1e-6 max(L) of d; the FP32 square and reach add relative errors
        // below 4e-7 and 1.2e-6, covered by the extra 1e-4 while R < 50
        // (a margin beyond every pair otherwise).
        // So (fl(R) + margin)^2 >= fl(d^2) for every kept pair, and
        // fl(d^2) < (fl(R) - margin)^2 only for pairs with d below R by more
        // than the FP64 keep rule's rounding: those are kept without it.
        // Only the pairs in the band between take the exact FP64 test.
        auto screen = [&](uint32_t t, const float4& qj, float qx, float qy, float qz) {
            const float fx = qx - qj.x, fy = qy - qj.y, fz = qz - qj.z;
            const float rs = qi.w + qj.w, rr = rs + margin;
            const float d2f = fx * fx + fy * fy + fz * fz;
            if (d2f > rr * rr) return;
            const float rl = rs - margin;
            s_q[nq++][tid] = t | (d2f < rl * fabsf(rl) ? kSurePair : 0u);
            if (!Together && nq == kNarrowQueue) work_off();
        };
        uint32_t t = 0, te = 0;
        float2 yz = make_float2(0.f, 0.f);
        if (Together) {
            constexpr int kGroup = 2;   // screens between two votes
            bool more = live;
            for (int k = -1; __any_sync(0xffffffffu, more);) {
                for (int r = 0; r < kGroup && more; ++r) {
                    if (t >= te) {
                        do {
                            if (++k == kNarrowRows) break;
                            t = s_t0[k][tid];
                            te = s_t1[k][tid];
                        } while (t >= te);
                        if (k == kNarrowRows) {
                            more = false;
                            break;
                        }
                        yz = s_yz[k][tid];
                    }
                    screen(t, p32s[t], qi.x, yz.x, yz.y);
                    ++t;
                }
                if (__any_sync(0xffffffffu, nq > kNarrowQueue - kGroup)) work_off();
            }
            if (!live) break;
        } else {
            for (int k = -1;;) {
                if (t >= te) {
                    do {
                        if (++k == kNarrowRows) break;
                        t = s_t0[k][tid];
                        te = s_t1[k][tid];
                    } while (t >= te);
                    if (k == kNarrowRows) break;
                    yz = s_yz[k][tid];
                }
                screen(t, p32s[t], qi.x, yz.x, yz.y);
                ++t;
            }
        }
        if (wrap_x && (cx == 0 || cx == d0 - 1)) {   // the images across x; within its own row only the one ahead
            const int xw = cx == 0 ? d0 - 1 : 0;
            const float qx = cx == 0 ? qi.x + g.Lf[0] : qi.x - g.Lf[0];
#pragma unroll 1
            for (int k = cx == 0 ? 1 : 0; k < kNarrowRows; ++k) {
                int z, y;
                float sy, sz;
                if (!axis_cell(cz + (k > 1), d2, g.periodic[2], g.Lf[2], z, sz) ||
                    !axis_cell(cy + (k > 1 ? k - 3 : k), d1, g.periodic[1], g.Lf[1], y, sy))
                    continue;
                const uint32_t row = ((uint32_t)z * (uint32_t)d1 + (uint32_t)y) * (uint32_t)d0 + (uint32_t)xw;
                for (uint32_t u = cs[row], ue = cs[row + 1]; u < ue; ++u) {
                    if (Together && nq == kNarrowQueue) work_off();
                    screen(u, p32s[u], qx, qi.y + sy, qi.z + sz);
                }
            }
        }
        work_off();
        double hi_ = -1.0;   // the exact hull of i, computed when a wall test needs it
        // walls: a conservative FP32 test of the signed distance (errors as
        // for the pairs, within wmargin), the exact FP64 test for the rest
        uint32_t wmask = 0;
        const int nwall = planes.count + planes.ncones + (V.batch ? 6 : 0);
        const float reach = qi.w + g.tauf + g.wmargin;
        for (int k = 0; k < nwall; ++k) {
            const int kc = k - planes.count;
            if (kc >= 0 && kc < planes.ncones) {   // cone (plain scenes only)
                if (cone_distance_f(g, kc, qi) > qi.w + g.tauf + g.cmargin) continue;
                double nrm[3], sd;
                const double4_32a pi = pos_r[i];
                if (!(hi_ >= 0.0)) hi_ = hull_of<Together>(H, i, pi.w);
                if (cone_distance(planes.cone[kc], pi, sd, nrm) && xsub(sd, pi.w) <= xadd(hi_, g.tau))
                    wmask |= 1u << k;
                continue;
            }
            float sdf;
            if (k < planes.count) {
                sdf = g.pn[k][0] * qi.x + g.pn[k][1] * qi.y + g.pn[k][2] * qi.z + g.pc[k];
            } else {
                const int f = k - planes.count, axis = f >> 1;
                const float q = axis == 0 ? qi.x : (axis == 1 ? qi.y : qi.z);
                const float* b = V.box32 + 6 * (int64_t)si;
                sdf = (f & 1) == 0 ? q - b[axis] : b[3 + axis] - q;
            }
            if (sdf > reach) continue;
            double nrm[3], c, sd, xi;
            uint32_t widx;
            wall_plane(planes, V, si, k, nrm, c, widx);
            const double4_32a pi = pos_r[i];
            if (!(hi_ >= 0.0)) hi_ = hull_of<Together>(H, i, pi.w);
            if (wall_kept(nrm, c, pi, hi_, g.tau, sd, xi)) wmask |= 1u << k;
        }
        wall_mask[i] = wmask;
    }
}

// The contacts' bodies: row i of the CSR holds (i, j) for the sorted partners
// j, then the walls in the order they were added.  A warp takes 32 bodies (in
// cell order) and spreads their sphere pairs over its lanes, one pair per
// lane and pass; the walls of a body stay with its own lane.
__global__ void k_write_ends(int64_t n, int64_t ccap, const uint32_t* __restrict__ svals,
                             const uint32_t* __restrict__ cand, const uint32_t* __restrict__ pair_cnt,
                             const uint32_t* __restrict__ wall_mask, const uint32_t* __restrict__ row_off,
                             int nplanes, int ncones, SceneView V, uint32_t* __restrict__ cj1,
                             uint32_t* __restrict__ cj2)
{
    const int lane = threadIdx.x & 31;
    const int64_t wstride = (int64_t)gridDim.x * blockDim.x;
    // warp-uniform trip count: every lane takes part in the shuffles
    for (int64_t s0 = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31u); s0 < n; s0 += wstride) {
        const int64_t s = s0 + lane;
        uint32_t i = 0, ns = 0, wm = 0, ro = 0;
        if (s < n) {
            i = svals[s];
            ns = min(pair_cnt[i], (uint32_t)kCandCap);
            wm = wall_mask[i];
            if ((ns | wm) != 0) ro = row_off[i];
        }
        uint32_t pre = ns;   // inclusive prefix of the pair counts over the lanes
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t v = __shfl_up_sync(0xffffffffu, pre, o);
            if (lane >= o) pre += v;
        }
        const uint32_t total = __shfl_sync(0xffffffffu, pre, 31);
        for (uint32_t base = 0; base < total; base += 32) {
            const uint32_t t = base + lane;
            // owner: the number of lanes whose pairs end at or before t
            int own = 0;
#pragma unroll
            for (int b = 16; b >= 1; b >>= 1) {
                const uint32_t v = __shfl_sync(0xffffffffu, pre, own + b - 1);
                if (v <= t) own += b;
            }
            own = own < 31 ? own : 31;
            const uint32_t i_o = __shfl_sync(0xffffffffu, i, own);
            const uint32_t ro_o = __shfl_sync(0xffffffffu, ro, own);
            const uint32_t end_o = __shfl_sync(0xffffffffu, pre, own);
            const uint32_t ns_o = __shfl_sync(0xffffffffu, ns, own);
            if (t >= total) continue;
            const uint32_t k = t - (end_o - ns_o);
            // the list holds its pairs as they were found: contact k goes to
            // the place of its partner in ascending order
            const uint32_t* list = cand + (int64_t)i_o * kCandCap;
            const uint32_t j = list[k];
            uint32_t rank = 0;
            for (uint32_t m = 0; m < ns_o; ++m) rank += list[m] < j ? 1u : 0u;
            const int64_t idx = (int64_t)ro_o + rank;
            if (idx >= ccap) continue;
            cj1[idx] = i_o;
            cj2[idx] = j;
        }
        if (wm == 0) continue;
        const uint32_t si = V.batch ? V.scene_of[i] : 0u;
        int64_t idx = (int64_t)ro + ns;
        for (uint32_t m = wm; m; m &= m - 1) {   // the walls k_narrow kept, in wall order
            const int k = __ffs(m) - 1;
            // planes and cones count from n, then six faces a scene
            const uint32_t w = (uint32_t)(V.n + k) + (k >= nplanes + ncones ? 6u * si : 0u);
            if (idx < ccap) {
                cj1[idx] = i;
                cj2[idx] = w;
            }
            ++idx;
        }
    }
}

// Normal, gap and levers of every contact, eq. (contactpos): a thread per
// contact.  A pair takes 35 FP64 instructions, each of which occupies its
// scheduler's FP64 unit for 64 cycles; that bounds the kernel (5.99M contacts
// 372 us, ncu, cold), so comparisons and the zeros of a lattice are read off
// the numbers' words.  Beside the colouring, on a stream of its own, it would
// spare a step of 2.75M contacts 100 us and one of 5.99M nothing.
__global__ void k_contact_geometry(DCount Cc, const double4_32a* __restrict__ pos_r,
                                   const uint32_t* __restrict__ cj1, const uint32_t* __restrict__ cj2, GridArgs g,
                                   const __grid_constant__ Planes planes, SceneView V, double4_32a* __restrict__ cgeo,
                                   double2* __restrict__ clev)
{
    const int64_t C = Cc.get();
    const double L0 = g.hi[0] - g.lo[0], L1 = g.hi[1] - g.lo[1], L2 = g.hi[2] - g.lo[2];
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < C; c += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t i = cj1[c], j = cj2[c];
        const double4_32a pi = pos_r[i];
        double nrm[3], xi, la, lb;
        if (j < (uint64_t)V.n) {
            const double4_32a pj = pos_r[j];
            const double dx3 = min_image(xsub(pi.x, pj.x), g.periodic[0], L0);
            const double dy3 = min_image(xsub(pi.y, pj.y), g.periodic[1], L1);
            const double dz3 = min_image(xsub(pi.z, pj.z), g.periodic[2], L2);
            // for spheres: n = (x_i - x_j)/d, the outward normal of S_j at its
            // point closest to x_i; xi = d - r_i - r_j
            const double d = pair_normal(dx3, dy3, dz3, nrm);
            xi = xsub(xsub(d, pi.w), pj.w);
            la = xsub(d, pj.w);
            lb = pj.w;
        } else {
            const uint32_t w = (uint32_t)(j - V.n);
            double sd, cc;
            if (w >= (uint32_t)planes.count && w < (uint32_t)(planes.count + planes.ncones)) {
                // the point of the cone's solid nearest to x_i is x_i - sd n:
                // a wall contact with xi = sd - r_i and l_i = -sd n
                cone_distance(planes.cone[w - planes.count], pi, sd, nrm);
                xi = xsub(sd, pi.w);
            } else {
                uint32_t widx;
                const uint32_t f = w - (uint32_t)planes.count;   // of a batch's boxes
                const bool face = w >= (uint32_t)planes.count;
                wall_plane(planes, V, face ? f / 6u : 0u, face ? planes.count + (int)(f % 6u) : (int)w, nrm, cc, widx);
                wall_kept(nrm, cc, pi, 0.0, g.tau, sd, xi);   // kept already: only sd and xi are used
            }
            la = sd;
            lb = 0.0;
        }
        cgeo[c] = make_double4_32a(nrm[0], nrm[1], nrm[2], xi);
        clev[c] = make_double2(la, lb);
    }
}

SceneView scene_view(const nbgs_scene* s)
{
    SceneView v;
    v.batch = s->batch ? 1 : 0;
    v.nplanes = s->planes.count;
    v.n = s->n;
    v.scene_of = s->scene_of;
    v.scene_off = s->scene_off;
    v.box = s->scene_box;
    v.box32 = s->scene_box32;
    v.mu = s->scene_mu;
    v.vref = s->scene_vref;
    v.body_of = s->composite ? s->mbody : nullptr;
    return v;
}

static GridArgs grid_args(const nbgs_scene* s)
{
    GridArgs g;
    for (int a = 0; a < 3; ++a) {
        g.lo[a] = s->prm.box_lo[a];
        g.hi[a] = s->prm.box_hi[a];
        g.periodic[a] = s->prm.periodic[a];
        g.dims_max[a] = s->dims_max[a];
    }
    g.r_max = s->r_max;
    g.dt = s->prm.dt;
    g.tau = s->prm.tau;
    double lmax = 0.0;
    for (int a = 0; a < 3; ++a) {
        g.Lf[a] = (float)(g.hi[a] - g.lo[a]);
        lmax = std::max(lmax, g.hi[a] - g.lo[a]);
    }
    g.margin = (float)(1e-4 + 1e-6 * lmax);
    g.pos_err = std::ldexp(lmax, -22);
    double cmax = 0.0;
    for (int k = 0; k < s->planes.count; ++k) {
        double off = -s->planes.c[k];
        for (int a = 0; a < 3; ++a) {
            g.pn[k][a] = (float)s->planes.n[k][a];
            off += s->planes.n[k][a] * g.lo[a];
        }
        g.pc[k] = (float)off;
        cmax = std::max(cmax, std::fabs(off));
    }
    g.tauf = (float)g.tau;
    g.wmargin = (float)(1e-4 + 4e-6 * (lmax + cmax));
    double amax = 0.0;
    for (int k = 0; k < s->planes.ncones; ++k) {
        const Cone& C = s->planes.cone[k];
        for (int a = 0; a < 3; ++a) {
            g.ca_apex[k][a] = (float)(C.apex[a] - g.lo[a]);
            g.ca_axis[k][a] = (float)C.axis[a];
            amax = std::max(amax, std::fabs(C.apex[a] - g.lo[a]));
        }
        g.ca_sc[k][0] = (float)C.sa;
        g.ca_sc[k][1] = (float)C.ca;
        g.ca_sc[k][2] = (float)C.s_o;
        g.ca_sc[k][3] = (float)C.s_t;
    }
    g.cmargin = (float)(1e-4 + 1e-5 * (lmax + amax));
    return g;
}

nbgs_status grow_contacts(nbgs_scene* s, int64_t need);  // api.cu

// Device-sized steps: the previous step's contact count, kept before the
// detection clears it; a count beyond the buffers sets the contact error bit.
__global__ void k_keep_count(DevInfo* info) { info->prev_contacts = info->n_contacts; }

__global__ void k_check_contacts(DevInfo* info, int64_t ccap)
{
    if ((int64_t)info->n_contacts > ccap) atomicOr(&info->err, kErrContacts);
}

static nbgs_status write_contacts(nbgs_scene* s, const GridArgs& g, DCount C)
{
    const int T = 256;
    k_write_ends<<<grid_for(s->n, T, 8, s->num_sms), T, 0, s->stream>>>(
        s->n, s->ccap, s->svals, s->cand, s->pair_cnt, s->wall_mask, s->row_off, s->planes.count, s->planes.ncones,
        scene_view(s), s->cj1, s->cj2);
    k_contact_geometry<<<grid_for(std::max<int64_t>(C.v, 1), T, 8, s->num_sms), T, 0, s->stream>>>(
        C, s->pos_r, s->cj1, s->cj2, g, s->planes, scene_view(s), s->cgeo, s->clev);
    return cuda_check(s, cudaGetLastError(), "detect");
}

// The limits of the detection, from the host's copy of the device's error
// bits: an ordinary step asks before it goes on, replayed ones when the host
// next looks.
nbgs_status check_detect_limits(nbgs_scene* s)
{
    const DevInfo& hi = *s->hinfo;
    if (hi.err & kErrGrid) return fail(s, NBGS_EINVAL, "detect: a periodic axis holds fewer than 3 grid cells");
    if (hi.err & kErrCand)
        return fail(s, NBGS_ECAPACITY, "detect: a body has " + std::to_string(hi.cand_need) +
                                           " hull neighbours above it (limit " + std::to_string(kCandCap) + ")");
    return NBGS_OK;
}

nbgs_status run_detect(nbgs_scene* s)
{
    const int64_t n = s->n;
    cudaStream_t st = s->stream;
    if (s->timing) cudaEventRecord(s->ev[0], st);
    // keep the previous step's contacts for the warm start
    if (s->prm.warm_start != NBGS_WARM_NONE && s->solved) {
        std::swap(s->row_off, s->prev_row_off);
        std::swap(s->cj2, s->prev_j2);
        std::swap(s->cworld, s->prev_P);
        s->prev_count = s->n_contacts;
        s->have_prev = true;
    }
    // otherwise the previous-step arrays keep what they hold: the contacts of
    // the last solved step, or of a restored checkpoint (nbgs_set_bodies
    // starts a new history)
    s->detected = s->coloured = s->solved = false;
    s->n_contacts = 0;
    s->sub_count = -1;
    if (s->device_sized) k_keep_count<<<1, 1, 0, st>>>(s->info);
    cudaMemsetAsync(s->info, 0, offsetof(DevInfo, cell_w), st);   // hmax, vmax
    cudaMemsetAsync(&s->info->n_contacts, 0, sizeof(uint32_t), st);
    if (n == 0) {
        cudaMemsetAsync(s->row_off, 0, sizeof(uint32_t), st);
        s->detected = true;
        return cuda_check(s, cudaGetLastError(), "detect");
    }
    const GridArgs g = grid_args(s);
    const int T = 256;
    const int gb = grid_for(n, T, 8, s->num_sms);
    if (s->batch) cudaMemsetAsync(s->scene_vmax, 0, s->n_scenes * sizeof(unsigned long long), st);
    if (s->composite) {
        if (s->fp32)
            k_member_update<float><<<gb, T, 0, st>>>(n, s->mbody, s->moff, s->bpos, s->bquat, (const float4*)s->bvel,
                                                     s->prm.dt, s->prm.tau, s->pos_r, s->hull, s->p32, g, s->info);
        else
            k_member_update<double><<<gb, T, 0, st>>>(n, s->mbody, s->moff, s->bpos, s->bquat,
                                                      (const double4_32a*)s->bvel, s->prm.dt, s->prm.tau, s->pos_r,
                                                      s->hull, s->p32, g, s->info);
    } else if (s->fp32)
        k_hull<float><<<gb, T, 0, st>>>(n, (const float4*)s->vel, s->pos_r, s->prm.dt, s->prm.tau, s->p32, g, s->info,
                                        s->scene_of, s->scene_vmax);
    else
        k_hull<double><<<gb, T, 0, st>>>(n, (const double4_32a*)s->vel, s->pos_r, s->prm.dt, s->prm.tau, s->p32, g,
                                         s->info, s->scene_of, s->scene_vmax);
    cudaMemsetAsync(s->cell_end, 0, (size_t)s->max_cells * sizeof(uint32_t), st);   // cell counts
    k_cell_keys<<<gb, T, 0, st>>>(n, s->p32, g, s->info, s->ckey, s->crank, s->cell_end);
    // first slot of every cell (empty ones included); cell_start[max_cells] = n
    nbgs_status rc = exclusive_scan_u32(s, s->cell_end, s->cell_start, s->max_cells, nullptr);
    if (rc != NBGS_OK) return rc;
    k_cell_scatter<<<gb, T, 0, st>>>(n, s->ckey, s->crank, s->cell_start, s->p32, s->svals, s->p32s);
    if (s->timing) s->phase_launches[0] += 5;
    cudaMemsetAsync(s->pair_cnt, 0, (size_t)n * sizeof(uint32_t), st);
    const HullView H{s->composite ? s->hull : nullptr, s->vel, s->fp32 ? 1 : 0, s->prm.dt, s->prm.tau};
    const bool together = s->composite && 2 * (int64_t)s->hinfo->n_contacts >= 3 * n;
    const int nb = grid_for(n, kNarrowThreads, 16, s->num_sms);
    if (together)
        k_narrow<true><<<nb, kNarrowThreads, 0, st>>>(n, s->svals, s->pos_r, H, s->p32s, s->cell_start, g, s->planes,
                                                      scene_view(s), s->info, s->cand, s->pair_cnt, s->wall_mask);
    else
        k_narrow<false><<<nb, kNarrowThreads, 0, st>>>(n, s->svals, s->pos_r, H, s->p32s, s->cell_start, g, s->planes,
                                                       scene_view(s), s->info, s->cand, s->pair_cnt, s->wall_mask);
    rc = exclusive_scan(s, ScanRows{s->pair_cnt, s->wall_mask}, s->row_off, DCount{n, nullptr}, &s->info->n_contacts);
    if (rc != NBGS_OK) return rc;
    if (s->timing) s->phase_launches[0] += 3;
    if (s->device_sized) {
        // no synchronisation: the buffers keep their capacity, an overflow
        // sets an error bit (the writes past it are skipped), and every
        // later kernel reads the count on the device
        k_check_contacts<<<1, 1, 0, st>>>(s->info, s->ccap);
        rc = write_contacts(s, g, contact_count(s));
        if (rc != NBGS_OK) return rc;
        if (s->timing) {
            s->phase_launches[0] += 4;
            cudaEventRecord(s->ev[1], st);
        }
        s->n_contacts = s->ccap;   // an upper bound; the count itself stays on the device
        s->detected = true;
        return cuda_check(s, cudaGetLastError(), "detect");
    }
    // one synchronisation per step: the contact count sizes everything after
    rc = cuda_check(s, cudaMemcpyAsync(s->hinfo, s->info, offsetof(DevInfo, rk_bits), cudaMemcpyDeviceToHost, st),
                    "detect: read info");
    if (rc != NBGS_OK) return rc;
    rc = cuda_check(s, cudaStreamSynchronize(st), "detect");
    if (rc != NBGS_OK) return rc;
    const DevInfo& hi = *s->hinfo;
    if (hi.err & kErrNaN) return fail(s, NBGS_ENAN, "detect: NaN or Inf in the velocities");
    rc = check_detect_limits(s);
    if (rc != NBGS_OK) return rc;
    const int64_t nc = hi.n_contacts;
    if (nc > s->ccap) {
        rc = grow_contacts(s, nc);
        if (rc != NBGS_OK) return rc;
    }
    s->n_contacts = nc;
    rc = write_contacts(s, g, DCount{nc, nullptr});
    if (rc != NBGS_OK) return rc;
    if (s->timing) {
        s->phase_launches[0] += 2;
        cudaEventRecord(s->ev[1], st);
    }
    s->detected = true;
    return cuda_check(s, cudaGetLastError(), "detect");
}

}  // namespace nbgs

namespace nbgs {
__global__ void k_pair_normals(int64_t n, const double* __restrict__ dvec, double* __restrict__ out)
{
    for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x) {
        double nrm[3];
        const double d = pair_normal(dvec[3 * k], dvec[3 * k + 1], dvec[3 * k + 2], nrm);
        out[4 * k] = nrm[0];
        out[4 * k + 1] = nrm[1];
        out[4 * k + 2] = nrm[2];
        out[4 * k + 3] = d;
    }
}
}  // namespace nbgs

extern "C" nbgs_status nbgs_pair_normals(int64_t n, const double* dvec, double* out, void* stream)
{
    using namespace nbgs;
    if (n < 0 || (n > 0 && (!dvec || !out))) return NBGS_EINVAL;
    if (n == 0) return NBGS_OK;
    int dev = 0, sms = 1;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    k_pair_normals<<<grid_for(n, 256, 8, sms), 256, 0, (cudaStream_t)stream>>>(n, dvec, out);
    return cudaGetLastError() == cudaSuccess ? NBGS_OK : NBGS_ECUDA;
}
