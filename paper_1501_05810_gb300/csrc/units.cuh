// units.cuh -- one sphere contact relaxed by L lanes of a warp on versioned
// body records (the dataflow sweeps, flow.cu).
//
// Unit<float, 2>: the even lane of a pair carries the linear, the odd lane
// the angular velocities of both bodies; both run the same instructions with
// their own coefficients, and three shuffles add up the relative velocity.  A
// lane loads and stores one 128-bit word per body, a pair a whole 32-byte
// sector, and nothing has to change places.
// Unit<double, 4>: lanes 0, 1, 2 carry the components x, y, z of all four
// velocities and solve for the n, t, o component of the impulse.  An FP64
// instruction occupies its scheduler's unit for 64 cycles however many lanes
// it serves, so in a small scene the number of instructions in a row is what
// a relaxation takes: about 40 against 100 with a lane per contact.
// Unit<double, 1>: a lane per contact, the fewest FP64 instructions per
// contact: for scenes that fill the FP64 units.
#pragma once

#include "relax.cuh"

namespace nbgs {

constexpr unsigned kFull = 0xffffffffu;

// 128-bit words of a versioned body: loads and stores of .b128 with relaxed
// gpu scope are single-copy atomic.
__device__ __forceinline__ uint4 ld_b128(const uint4* p)
{
    unsigned long long lo, hi;
    asm volatile("{\n\t.reg .b128 t;\n\tld.relaxed.gpu.global.b128 t, [%2];\n\tmov.b128 {%0, %1}, t;\n\t}"
                 : "=l"(lo), "=l"(hi)
                 : "l"(p)
                 : "memory");
    return make_uint4((uint32_t)lo, (uint32_t)(lo >> 32), (uint32_t)hi, (uint32_t)(hi >> 32));
}

__device__ __forceinline__ void st_b128(uint4* p, const uint4& v)
{
    const unsigned long long lo = ((unsigned long long)v.y << 32) | v.x, hi = ((unsigned long long)v.w << 32) | v.z;
    asm volatile("{\n\t.reg .b128 t;\n\tmov.b128 t, {%1, %2};\n\tst.relaxed.gpu.global.b128 [%0], t;\n\t}" ::"l"(p),
                 "l"(lo), "l"(hi)
                 : "memory");
}

__device__ __forceinline__ double join(uint32_t lo, uint32_t hi) { return __hiloint2double((int)hi, (int)lo); }
__device__ __forceinline__ uint32_t lo32(double x) { return (uint32_t)__double2loint(x); }
__device__ __forceinline__ uint32_t hi32(double x) { return (uint32_t)__double2hiint(x); }

// A body's record.  FP32, two words: (v, tag), (w, tag).  FP64, four: (v_j,
// low half of w_j, tag) for j = x, y, z, and the high halves of w with the tag.
template <class R> struct Words;
template <> struct Words<float> { static constexpr int N = 2; };
template <> struct Words<double> { static constexpr int N = 4; };

__device__ __forceinline__ void pack_body(uint4* q, uint32_t tag, const float4& v, const float4& w)
{
    st_b128(q, make_uint4(__float_as_uint(v.x), __float_as_uint(v.y), __float_as_uint(v.z), tag));
    st_b128(q + 1, make_uint4(__float_as_uint(w.x), __float_as_uint(w.y), __float_as_uint(w.z), tag));
}
__device__ __forceinline__ void pack_body(uint4* q, uint32_t tag, const double4_32a& v, const double4_32a& w)
{
    st_b128(q, make_uint4(lo32(v.x), hi32(v.x), lo32(w.x), tag));
    st_b128(q + 1, make_uint4(lo32(v.y), hi32(v.y), lo32(w.y), tag));
    st_b128(q + 2, make_uint4(lo32(v.z), hi32(v.z), lo32(w.z), tag));
    st_b128(q + 3, make_uint4(hi32(w.x), hi32(w.y), hi32(w.z), tag));
}
__device__ __forceinline__ void load_body(const uint4* q, float4& v, float4& w, uint32_t* tags)
{
    const uint4 a = ld_b128(q), b = ld_b128(q + 1);
    v = make_float4(__uint_as_float(a.x), __uint_as_float(a.y), __uint_as_float(a.z), 0.f);
    w = make_float4(__uint_as_float(b.x), __uint_as_float(b.y), __uint_as_float(b.z), 0.f);
    tags[0] = a.w;
    tags[1] = b.w;
}
__device__ __forceinline__ void load_body(const uint4* q, double4_32a& v, double4_32a& w, uint32_t* tags)
{
    const uint4 a = ld_b128(q), b = ld_b128(q + 1), c = ld_b128(q + 2), d = ld_b128(q + 3);
    v = make_double4_32a(join(a.x, a.y), join(b.x, b.y), join(c.x, c.y), 0.0);
    w = make_double4_32a(join(a.z, d.x), join(b.z, d.y), join(c.z, d.z), 0.0);
    tags[0] = a.w;
    tags[1] = b.w;
    tags[2] = c.w;
    tags[3] = d.w;
}

// What a contact needs besides its record does not change during a solve.
__device__ __forceinline__ SweepPre<float> ld_pre(const SweepPre<float>* p)
{
    SweepPre<float> x;
    asm("ld.global.nc.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
        : "=f"(x.m.x), "=f"(x.m.y), "=f"(x.m.z), "=f"(x.m.w), "=f"(x.w.x), "=f"(x.w.y), "=f"(x.w.z), "=f"(x.w.w)
        : "l"(p));
    return x;
}
__device__ __forceinline__ SweepPre<double> ld_pre(const SweepPre<double>* p)
{
    SweepPre<double> x;
    asm("ld.global.nc.v4.f64 {%0,%1,%2,%3}, [%4];" : "=d"(x.m.x), "=d"(x.m.y), "=d"(x.m.z), "=d"(x.m.w) : "l"(p));
    asm("ld.global.nc.v4.f64 {%0,%1,%2,%3}, [%4];"
        : "=d"(x.w.x), "=d"(x.w.y), "=d"(x.w.z), "=d"(x.w.w)
        : "l"(reinterpret_cast<const char*>(p) + 32));
    return x;
}

// First tile of every colour (tw contacts per tile), and the colour offsets,
// for the block; every thread takes part.
__device__ __forceinline__ void tile_offsets(const uint32_t* col_off, int ncol, uint32_t tw, uint32_t* s_off,
                                             uint32_t* s_tile)
{
    for (int c = threadIdx.x; c <= ncol; c += blockDim.x) s_off[c] = col_off[c];
    __syncthreads();
    if (threadIdx.x < 32) {
        const int lane = threadIdx.x;
        uint32_t carry = 0;
        for (int c0 = 0; c0 < ncol; c0 += 32) {
            const int c = c0 + lane;
            uint32_t v = c < ncol ? (s_off[c + 1] - s_off[c] + tw - 1) / tw : 0u;
            const uint32_t own = v;
            for (int o = 1; o < 32; o <<= 1) {
                const uint32_t y = __shfl_up_sync(kFull, v, o);
                if (lane >= o) v += y;
            }
            if (c < ncol) s_tile[c] = carry + v - own;
            carry += __shfl_sync(kFull, v, 31);
        }
        if (lane == 0) s_tile[ncol] = carry;
    }
    __syncthreads();
}

template <class R, int L> struct Unit;

// a b + c d + e f and a b - c d with the operations fused as the compiler
// fuses these expressions in relax_bodies.
__device__ __forceinline__ float dot3(float a, float b, float c, float d, float e, float f)
{
    return fmaf(e, f, fmaf(a, b, __fmul_rn(c, d)));
}
__device__ __forceinline__ float cross1(float a, float b, float c, float d) { return fmaf(a, b, -__fmul_rn(c, d)); }

// The constant part of an FP32 contact, and the relaxed impulse for a relative
// velocity u: every operation rounded as in relax_bodies, so that the results
// are those of the other sweep kernels bit for bit.
struct Contact32 {
    float nx, ny, nz, tx, ty, tz, ox, oy, la, lb, bias, wn, wt, rwn, rwt;   // oz = -ny
    bool hasb, moves, fast;

    __device__ __forceinline__ void set(const SweepRec<float>& rr, const SweepPre<float>& x, uint32_t& ia, uint32_t& ib,
                                        uint32_t n)
    {
        decode<float>(rr, ia, ib, la, lb, nx, ny, nz, bias);
        // tangent_basis with its factor stored
        const float sign = copysignf(1.f, nz), f = x.w.w, m = __fmul_rn(__fmul_rn(nx, ny), f);
        const float sx = __fmul_rn(sign, nx);
        tx = fmaf(__fmul_rn(sx, nx), f, 1.f);
        ty = __fmul_rn(sign, m);
        tz = -sx;
        ox = m;
        oy = fmaf(__fmul_rn(ny, ny), f, sign);
        wn = x.m.x + x.m.y;
        wt = x.w.x;
        rwn = x.w.y;
        rwt = x.w.z;
        hasb = ib < n;
        moves = wn > 0.f;   // both masses infinite: nothing can move
        fast = recip_ok(wn, wt) || !moves;
        if (!hasb) ib = ia;   // a wall: any record will do, nothing of it is used
    }

    // the change (dn, dt, do) of the impulse pp for relative velocity u; p
    // the new one
    __device__ __forceinline__ void solve(float ux, float uy, float uz, float mu, float omega, const float4& pp, float3& p,
                                          float& dn, float& dt, float& do_) const
    {
        const float un = dot3(nx, ux, ny, uy, nz, uz);
        const float ut = dot3(tx, ux, ty, uy, tz, uz);
        const float uo = dot3(ox, ux, oy, uy, -ny, uz);
        const float bn = __fadd_rn(fmaf(-wn, pp.x, un), bias);
        const float bt = fmaf(-wt, pp.y, ut);
        const float bo = fmaf(-wt, pp.z, uo);
        float yn = quotient(-bn, wn, rwn), yt = quotient(-bt, wt, rwt), yo = quotient(-bo, wt, rwt);
        if (__any_sync(kFull, !fast)) {   // masses beyond the reciprocals' range
            if (!fast) {
                yn = -bn / wn;
                yt = -bt / wt;
                yo = -bo / wt;
            }
        }
        yn = clamp0(yn);
        const float lim = __fmul_rn(mu, yn);
        const float len2 = fmaf(yt, yt, __fmul_rn(yo, yo));
        if (len2 > __fmul_rn(lim, lim)) {
            const float sc = __fdiv_rn(lim, __fsqrt_rn(len2));
            yt = __fmul_rn(yt, sc);
            yo = __fmul_rn(yo, sc);
        }
        if (omega != 1.f) {
            const float om1 = 1.f - omega;
            yn = fmaf(om1, pp.x, __fmul_rn(omega, yn));
            yt = fmaf(om1, pp.y, __fmul_rn(omega, yt));
            yo = fmaf(om1, pp.z, __fmul_rn(omega, yo));
        }
        dn = __fsub_rn(yn, pp.x);
        dt = __fsub_rn(yt, pp.y);
        do_ = __fsub_rn(yo, pp.z);
        p = make_float3(yn, yt, yo);
    }

    // world impulse change and its torque arm
    __device__ __forceinline__ void world(float dn, float dt, float do_, float3& P, float3& q) const
    {
        P.x = dot3(dn, nx, dt, tx, do_, ox);
        P.y = dot3(dn, ny, dt, ty, do_, oy);
        P.z = dot3(dn, nz, dt, tz, do_, -ny);
        q.x = cross1(ny, P.z, nz, P.y);
        q.y = cross1(nz, P.x, nx, P.z);
        q.z = cross1(nx, P.y, ny, P.x);
    }

    __device__ __forceinline__ float residual(float dn, float dt, float do_) const
    {
        const float r1 = __fmul_rn(wn, dn), r2 = __fmul_rn(wt, dt), r3 = __fmul_rn(wt, do_);
        return dot3(r1, r1, r2, r2, r3, r3);
    }
};

template <> struct Unit<float, 2> {
    Contact32 C;
    float o1, o2;                   // factors of the change of this lane's halves
    float4 pp;
    uint32_t qa, qb;                // this lane's words of the two bodies
    bool hasb;
    uint4 xa, xb;                   // their contents
    float dn, dt, do_;

    __device__ __forceinline__ static bool odd() { return (threadIdx.x & 1u) != 0u; }

    __device__ __forceinline__ void take(const SweepRec<float>& rr, const SweepPre<float>& x, const float4& p, uint32_t n)
    {
        uint32_t ia, ib;
        C.set(rr, x, ia, ib, n);
        hasb = C.hasb;
        o1 = odd() ? -x.m.z : x.m.x;
        o2 = odd() ? -x.m.w : -x.m.y;
        pp = p;
        const uint32_t h = threadIdx.x & 1u;
        qa = 2u * ia + h;
        qb = 2u * ib + h;
    }
    __device__ __forceinline__ void idle(uint32_t q)
    {
        qa = qb = q;
        hasb = C.moves = false;
        C.fast = true;
    }

    __device__ __forceinline__ void load(const uint4* tv)
    {
        xa = ld_b128(tv + qa);
        xb = ld_b128(tv + qb);
    }
    // whether the versions loaded are those wanted (ma, mb: all ones for a
    // body with versions, else 0)
    __device__ __forceinline__ bool ready(uint32_t ma, uint32_t mb, uint32_t ta, uint32_t tb) const
    {
        return (((xa.w ^ ta) & ma) | ((xb.w ^ tb) & mb)) == 0u;
    }
    __device__ __forceinline__ void store(uint4* tv, bool va, bool vb, uint32_t ta, uint32_t tb)
    {
        xa.w = ta;
        xb.w = tb;
        if (va) st_b128(tv + qa, xa);
        if (vb) st_b128(tv + qb, xb);
    }
    __device__ __forceinline__ void save(float4* p) const
    {
        if (!odd()) *p = pp;
    }

    // Every lane of the warp takes part (live: its contact is relaxed); the
    // velocities are updated, residual() gives r_j^2 afterwards.
    template <bool apply_only>
    __device__ __forceinline__ void relax(bool live, float mu, float omega)
    {
        const float ax = __uint_as_float(xa.x), ay = __uint_as_float(xa.y), az = __uint_as_float(xa.z);
        float bx = __uint_as_float(xb.x), by = __uint_as_float(xb.y), bz = __uint_as_float(xb.z);
        bx = C.hasb ? bx : 0.f;
        by = C.hasb ? by : 0.f;
        bz = C.hasb ? bz : 0.f;
        const bool act = live && C.moves;
        if (apply_only) {
            dn = pp.x;
            dt = pp.y;
            do_ = pp.z;
        } else {
            // w x n on the odd lane, handed to the even one, which solves
            float cax = cross1(ay, C.nz, az, C.ny), cay = cross1(az, C.nx, ax, C.nz), caz = cross1(ax, C.ny, ay, C.nx);
            float cbx = cross1(by, C.nz, bz, C.ny), cby = cross1(bz, C.nx, bx, C.nz), cbz = cross1(bx, C.ny, by, C.nx);
            cax = __shfl_xor_sync(kFull, cax, 1);
            cay = __shfl_xor_sync(kFull, cay, 1);
            caz = __shfl_xor_sync(kFull, caz, 1);
            cbx = __shfl_xor_sync(kFull, cbx, 1);
            cby = __shfl_xor_sync(kFull, cby, 1);
            cbz = __shfl_xor_sync(kFull, cbz, 1);
            const float ux = __fsub_rn(fmaf(-C.la, cax, ax), fmaf(C.lb, cbx, bx));
            const float uy = __fsub_rn(fmaf(-C.la, cay, ay), fmaf(C.lb, cby, by));
            const float uz = __fsub_rn(fmaf(-C.la, caz, az), fmaf(C.lb, cbz, bz));
            float3 p;
            C.solve(ux, uy, uz, mu, omega, pp, p, dn, dt, do_);
            if (act) {
                pp.x = p.x;
                pp.y = p.y;
                pp.z = p.z;
            }
            const float rn = __shfl_xor_sync(kFull, dn, 1), rt = __shfl_xor_sync(kFull, dt, 1),
                        ro = __shfl_xor_sync(kFull, do_, 1);
            dn = odd() ? rn : dn;
            dt = odd() ? rt : dt;
            do_ = odd() ? ro : do_;
        }
        dn = act ? dn : 0.f;
        dt = act ? dt : 0.f;
        do_ = act ? do_ : 0.f;
        float3 P, q;
        C.world(dn, dt, do_, P, q);
        const float X = odd() ? q.x : P.x, Y = odd() ? q.y : P.y, Z = odd() ? q.z : P.z;
        xa.x = __float_as_uint(fmaf(o1, X, ax));
        xa.y = __float_as_uint(fmaf(o1, Y, ay));
        xa.z = __float_as_uint(fmaf(o1, Z, az));
        xb.x = __float_as_uint(fmaf(o2, X, bx));
        xb.y = __float_as_uint(fmaf(o2, Y, by));
        xb.z = __float_as_uint(fmaf(o2, Z, bz));
    }
    __device__ __forceinline__ float residual() const { return C.residual(dn, dt, do_); }
};

template <> struct Unit<float, 1> {
    Contact32 C;
    float ima, imb, ka, kb;
    float4 pp;
    uint32_t qa, qb;                // first words of the two bodies
    bool hasb;
    uint4 av, aw, bv, bw;           // the bodies: (v, tag), (w, tag)
    float dn, dt, do_;

    __device__ __forceinline__ static bool odd() { return (threadIdx.x & 1u) != 0u; }
    __device__ __forceinline__ static uint4 swap(const uint4& v)
    {
        return make_uint4(__shfl_xor_sync(kFull, v.x, 1), __shfl_xor_sync(kFull, v.y, 1),
                          __shfl_xor_sync(kFull, v.z, 1), __shfl_xor_sync(kFull, v.w, 1));
    }
    __device__ __forceinline__ static uint4 pick(bool c, const uint4& a, const uint4& b)
    {
        return make_uint4(c ? a.x : b.x, c ? a.y : b.y, c ? a.z : b.z, c ? a.w : b.w);
    }

    __device__ __forceinline__ void take(const SweepRec<float>& rr, const SweepPre<float>& x, const float4& p, uint32_t n)
    {
        uint32_t ia, ib;
        C.set(rr, x, ia, ib, n);
        hasb = C.hasb;
        ima = x.m.x;
        imb = x.m.y;
        ka = x.m.z;
        kb = x.m.w;
        pp = p;
        qa = 2u * ia;
        qb = 2u * ib;
    }
    __device__ __forceinline__ void idle(uint32_t q)
    {
        qa = qb = q;
        hasb = C.moves = false;
        C.fast = true;
    }

    // Lanes 2i and 2i + 1 fetch the two words of one body after the other and
    // swap them, so that every access of a pair is a whole 32-byte sector.
    __device__ __forceinline__ void load(const uint4* tv)
    {
        const bool o = odd();
        const uint32_t a2 = __shfl_xor_sync(kFull, qa, 1), b2 = __shfl_xor_sync(kFull, qb, 1);
        const uint4* t = tv + (o ? 1 : 0);
        const uint4 x0 = ld_b128(t + (o ? a2 : qa)), x1 = ld_b128(t + (o ? qa : a2));
        const uint4 y0 = ld_b128(t + (o ? b2 : qb)), y1 = ld_b128(t + (o ? qb : b2));
        const uint4 xr = swap(pick(o, x0, x1)), yr = swap(pick(o, y0, y1));
        av = pick(o, xr, x0);
        aw = pick(o, x1, xr);
        bv = pick(o, yr, y0);
        bw = pick(o, y1, yr);
    }
    __device__ __forceinline__ bool ready(uint32_t ma, uint32_t mb, uint32_t ta, uint32_t tb) const
    {
        return (((av.w ^ ta) & ma) | ((aw.w ^ ta) & ma) | ((bv.w ^ tb) & mb) | ((bw.w ^ tb) & mb)) == 0u;
    }
    __device__ __forceinline__ void store(uint4* tv, bool va, bool vb, uint32_t ta, uint32_t tb)
    {
        const bool o = odd();
        const uint32_t a2 = __shfl_xor_sync(kFull, qa, 1), b2 = __shfl_xor_sync(kFull, qb, 1);
        const uint32_t w = (va ? 1u : 0u) | (vb ? 2u : 0u), w2 = __shfl_xor_sync(kFull, w, 1);
        av.w = aw.w = ta;
        bv.w = bw.w = tb;
        const uint4 ar = swap(pick(o, av, aw)), br = swap(pick(o, bv, bw));
        uint4* t = tv + (o ? 1 : 0);
        const uint32_t we = o ? w2 : w, wo = o ? w : w2;   // what the even and the odd lane want stored
        if (we & 1u) st_b128(t + (o ? a2 : qa), pick(o, ar, av));
        if (wo & 1u) st_b128(t + (o ? qa : a2), pick(o, aw, ar));
        if (we & 2u) st_b128(t + (o ? b2 : qb), pick(o, br, bv));
        if (wo & 2u) st_b128(t + (o ? qb : b2), pick(o, bw, br));
    }
    __device__ __forceinline__ void save(float4* p) const { *p = pp; }

    template <bool apply_only>
    __device__ __forceinline__ void relax(bool live, float mu, float omega)
    {
        float vax = __uint_as_float(av.x), vay = __uint_as_float(av.y), vaz = __uint_as_float(av.z);
        float wax = __uint_as_float(aw.x), way = __uint_as_float(aw.y), waz = __uint_as_float(aw.z);
        float vbx = __uint_as_float(bv.x), vby = __uint_as_float(bv.y), vbz = __uint_as_float(bv.z);
        float wbx = __uint_as_float(bw.x), wby = __uint_as_float(bw.y), wbz = __uint_as_float(bw.z);
        if (!C.hasb) vbx = vby = vbz = wbx = wby = wbz = 0.f;
        const bool act = live && C.moves;
        if (apply_only) {
            dn = pp.x;
            dt = pp.y;
            do_ = pp.z;
        } else {
            const float cax = cross1(way, C.nz, waz, C.ny), cay = cross1(waz, C.nx, wax, C.nz),
                        caz = cross1(wax, C.ny, way, C.nx);
            const float cbx = cross1(wby, C.nz, wbz, C.ny), cby = cross1(wbz, C.nx, wbx, C.nz),
                        cbz = cross1(wbx, C.ny, wby, C.nx);
            const float ux = __fsub_rn(fmaf(-C.la, cax, vax), fmaf(C.lb, cbx, vbx));
            const float uy = __fsub_rn(fmaf(-C.la, cay, vay), fmaf(C.lb, cby, vby));
            const float uz = __fsub_rn(fmaf(-C.la, caz, vaz), fmaf(C.lb, cbz, vbz));
            float3 p;
            C.solve(ux, uy, uz, mu, omega, pp, p, dn, dt, do_);
            if (act) {
                pp.x = p.x;
                pp.y = p.y;
                pp.z = p.z;
            }
        }
        dn = act ? dn : 0.f;
        dt = act ? dt : 0.f;
        do_ = act ? do_ : 0.f;
        float3 P, q;
        C.world(dn, dt, do_, P, q);
        av.x = __float_as_uint(fmaf(ima, P.x, vax));
        av.y = __float_as_uint(fmaf(ima, P.y, vay));
        av.z = __float_as_uint(fmaf(ima, P.z, vaz));
        aw.x = __float_as_uint(fmaf(-ka, q.x, wax));
        aw.y = __float_as_uint(fmaf(-ka, q.y, way));
        aw.z = __float_as_uint(fmaf(-ka, q.z, waz));
        bv.x = __float_as_uint(fmaf(-imb, P.x, vbx));
        bv.y = __float_as_uint(fmaf(-imb, P.y, vby));
        bv.z = __float_as_uint(fmaf(-imb, P.z, vbz));
        bw.x = __float_as_uint(fmaf(-kb, q.x, wbx));
        bw.y = __float_as_uint(fmaf(-kb, q.y, wby));
        bw.z = __float_as_uint(fmaf(-kb, q.z, wbz));
    }
    __device__ __forceinline__ float residual() const { return C.residual(dn, dt, do_); }
};

template <> struct Unit<double, 1> {
    double nx, ny, nz, tx, ty, tz, ox, oy, oz, la, lb, bias, ima, imb, ka, kb, wn, wt, rwn, rwt;
    double4_32a pp;
    uint32_t qa, qb;
    bool hasb, fast;
    double4_32a va, wa, vb, wb;
    uint32_t tags[2][4];

    __device__ __forceinline__ void take(const SweepRec<double>& rr, const SweepPre<double>& x, const double4_32a& p,
                                         uint32_t n)
    {
        uint32_t ia, ib;
        decode<double>(rr, ia, ib, la, lb, nx, ny, nz, bias);
        const double sign = copysign(1.0, nz), f = rr.nz_.y;   // tangent_basis with its factor stored
        const double m = nx * ny * f, sx = __hiloint2double(__double2hiint(nx) ^ (int)(hi32(sign) & 0x80000000u),
                                                            __double2loint(nx));
        tx = 1.0 + sx * nx * f;
        ty = __hiloint2double(__double2hiint(m) ^ (int)(hi32(sign) & 0x80000000u), __double2loint(m));
        tz = -sx;
        ox = m;
        oy = sign + ny * ny * f;
        oz = -ny;
        ima = x.m.x;
        imb = x.m.y;
        ka = x.m.z;
        kb = x.m.w;
        wn = x.w.x;
        wt = x.w.y;
        rwn = x.w.z;
        rwt = x.w.w;
        fast = recip_ok(wn, wt);
        hasb = ib < n;
        pp = p;
        if (!hasb) ib = ia;
        qa = 4u * ia;
        qb = 4u * ib;
    }
    __device__ __forceinline__ void idle(uint32_t q)
    {
        qa = qb = q;
        hasb = false;
        wn = 0.0;
    }
    __device__ __forceinline__ void load(const uint4* tv)
    {
        load_body(tv + qa, va, wa, tags[0]);
        load_body(tv + qb, vb, wb, tags[1]);
        if (!hasb) vb.x = vb.y = vb.z = 0.0;
    }
    __device__ __forceinline__ bool ready(uint32_t ma, uint32_t mb, uint32_t ta, uint32_t tb) const
    {
        uint32_t d = 0u;
#pragma unroll
        for (int j = 0; j < 4; ++j) d |= ((tags[0][j] ^ ta) & ma) | ((tags[1][j] ^ tb) & mb);
        return d == 0u;
    }
    __device__ __forceinline__ void store(uint4* tv, bool ha, bool hb, uint32_t ta, uint32_t tb) const
    {
        if (ha) pack_body(tv + qa, ta, va, wa);
        if (hb) pack_body(tv + qb, tb, vb, wb);
    }

    __device__ __forceinline__ void save(double4_32a* p) const { st_d4(p, pp); }

    double dn, dt, do_;
    template <bool apply_only>
    __device__ __forceinline__ void relax(bool live, double mu, double omega)
    {
        dn = dt = do_ = 0.0;
        if (!live || !above(wn, 0.0)) return;
        if (apply_only) {
            dn = pp.x;
            dt = pp.y;
            do_ = pp.z;
        } else {
            const double dx = va.x - vb.x, dy = va.y - vb.y, dz = va.z - vb.z;
            const double sx = la * wa.x + lb * wb.x, sy = la * wa.y + lb * wb.y, sz = la * wa.z + lb * wb.z;
            const double un = nx * dx + ny * dy + nz * dz;
            const double ut = tx * dx + ty * dy + tz * dz - ox * sx - oy * sy - oz * sz;
            const double uo = ox * dx + oy * dy + oz * dz + tx * sx + ty * sy + tz * sz;
            const double bn = un - wn * pp.x + bias, bt = ut - wt * pp.y, bo = uo - wt * pp.z;
            double yn, yt, yo;
            if (fast) {
                yn = quotient(-bn, wn, rwn);
                yt = quotient(-bt, wt, rwt);
                yo = quotient(-bo, wt, rwt);
            } else {
                yn = -bn / wn;
                yt = -bt / wt;
                yo = -bo / wt;
            }
            yn = clamp0(yn);
            const double lim = mu * yn, len2 = yt * yt + yo * yo;
            if (beyond(len2, lim * lim)) {
                const double sc = slide_scale(lim, len2);
                yt *= sc;
                yo *= sc;
            }
            if (omega != 1.0) {
                const double om1 = 1.0 - omega;
                yn = omega * yn + om1 * pp.x;
                yt = omega * yt + om1 * pp.y;
                yo = omega * yo + om1 * pp.z;
            }
            dn = yn - pp.x;
            dt = yt - pp.y;
            do_ = yo - pp.z;
            pp.x = yn;
            pp.y = yt;
            pp.z = yo;
        }
        const double Px = dn * nx + dt * tx + do_ * ox, Py = dn * ny + dt * ty + do_ * oy,
                     Pz = dn * nz + dt * tz + do_ * oz;
        const double qx = dt * ox - do_ * tx, qy = dt * oy - do_ * ty, qz = dt * oz - do_ * tz;
        va.x += ima * Px;
        va.y += ima * Py;
        va.z += ima * Pz;
        wa.x -= ka * qx;
        wa.y -= ka * qy;
        wa.z -= ka * qz;
        vb.x -= imb * Px;
        vb.y -= imb * Py;
        vb.z -= imb * Pz;
        wb.x -= kb * qx;
        wb.y -= kb * qy;
        wb.z -= kb * qz;
    }
    __device__ __forceinline__ double residual() const
    {
        const double r1 = wn * dn, r2 = wt * dt, r3 = wt * do_;
        return r1 * r1 + r2 * r2 + r3 * r3;
    }
};

template <> struct Unit<double, 4> {
    double n_, t_, o_;                  // component j of the frame (j = lane % 4; lane 3 idles along)
    double la, lb, ima, imb, ka, kb;
    double w, rw, bias, p;              // of the impulse component this lane solves for
    double4_32a pp;
    uint32_t qa, qb;
    bool hasb, fast;
    uint4 x, y;
    double va, wa, vb, wb, r;

    __device__ __forceinline__ static uint32_t sub() { return threadIdx.x & 3u; }
    __device__ __forceinline__ static double pick3(double x, double y, double z)
    {
        const uint32_t j = sub();
        return j == 0u ? x : (j == 1u ? y : z);
    }
    __device__ __forceinline__ static double from(double x, uint32_t j)   // lane j of the unit
    {
        return __shfl_sync(kFull, x, (int)j, 4);
    }

    __device__ __forceinline__ void take(const SweepRec<double>& rr, const SweepPre<double>& x, const double4_32a& q,
                                         uint32_t n)
    {
        uint32_t ia, ib;
        double nx, ny, nz, bi;
        decode<double>(rr, ia, ib, la, lb, nx, ny, nz, bi);
        const double sign = copysign(1.0, nz), fb = rr.nz_.y;
        const double m = nx * ny * fb;
        n_ = pick3(nx, ny, nz);
        t_ = pick3(1.0 + sign * nx * nx * fb, sign * m, -sign * nx);
        o_ = pick3(m, sign + ny * ny * fb, -ny);
        ima = x.m.x;
        imb = x.m.y;
        ka = x.m.z;
        kb = x.m.w;
        const bool first = sub() == 0u;
        w = first ? x.w.x : x.w.y;
        rw = first ? x.w.z : x.w.w;
        fast = recip_ok(x.w.x, x.w.y);
        bias = first ? bi : 0.0;
        hasb = ib < n;
        pp = q;
        p = pick3(q.x, q.y, q.z);
        if (!hasb) ib = ia;
        qa = 4u * ia + sub();
        qb = 4u * ib + sub();
    }
    __device__ __forceinline__ void idle(uint32_t q)
    {
        qa = qb = q;
        hasb = false;
        w = 0.0;
    }
    __device__ __forceinline__ void load(const uint4* tv)
    {
        x = ld_b128(tv + qa);
        y = ld_b128(tv + qb);
    }
    __device__ __forceinline__ bool ready(uint32_t ma, uint32_t mb, uint32_t ta, uint32_t tb) const
    {
        return (((x.w ^ ta) & ma) | ((y.w ^ tb) & mb)) == 0u;
    }
    __device__ __forceinline__ void store(uint4* tv, bool ha, bool hb, uint32_t ta, uint32_t tb) const
    {
        const uint32_t j = sub();
        const uint32_t ah = hi32(wa), bh = hi32(wb);
        const uint32_t a0 = __shfl_sync(kFull, ah, 0, 4), a1 = __shfl_sync(kFull, ah, 1, 4),
                       a2 = __shfl_sync(kFull, ah, 2, 4);
        const uint32_t b0 = __shfl_sync(kFull, bh, 0, 4), b1 = __shfl_sync(kFull, bh, 1, 4),
                       b2 = __shfl_sync(kFull, bh, 2, 4);
        if (ha) st_b128(tv + qa, j == 3u ? make_uint4(a0, a1, a2, ta) : make_uint4(lo32(va), hi32(va), lo32(wa), ta));
        if (hb) st_b128(tv + qb, j == 3u ? make_uint4(b0, b1, b2, tb) : make_uint4(lo32(vb), hi32(vb), lo32(wb), tb));
    }

    __device__ __forceinline__ void save(double4_32a* q) const
    {
        if (sub() < 3u) reinterpret_cast<double*>(q)[sub()] = p;
    }

    template <bool apply_only>
    __device__ __forceinline__ void relax(bool live, double mu, double omega)
    {
        const uint32_t j = sub();
        va = join(x.x, x.y);
        vb = hasb ? join(y.x, y.y) : 0.0;
        // the high halves of w come from lane 3
        const uint32_t a0 = __shfl_sync(kFull, x.x, 3, 4), a1 = __shfl_sync(kFull, x.y, 3, 4),
                       a2 = __shfl_sync(kFull, x.z, 3, 4);
        const uint32_t b0 = __shfl_sync(kFull, y.x, 3, 4), b1 = __shfl_sync(kFull, y.y, 3, 4),
                       b2 = __shfl_sync(kFull, y.z, 3, 4);
        wa = join(x.z, j == 0u ? a0 : (j == 1u ? a1 : a2));
        wb = join(y.z, j == 0u ? b0 : (j == 1u ? b1 : b2));
        const double wn = from(w, 0);
        const bool moves = live && above(wn, 0.0);
        double d;
        if (apply_only) {
            d = p;
        } else {
            const double dv = va - vb, s = la * wa + lb * wb;
            // partial sums of the three components of u, added up over the
            // lanes so that lane j ends with component j
            const double A0 = n_ * dv, A1 = t_ * dv - o_ * s, A2 = o_ * dv + t_ * s;
            const uint32_t nxt = j == 2u ? 0u : j + 1u, prv = j == 0u ? 2u : j - 1u;   // lane 3: any
            const double u = pick3(A0, A1, A2) + __shfl_sync(kFull, pick3(A2, A0, A1), (int)(nxt & 3u), 4) +
                             __shfl_sync(kFull, pick3(A1, A2, A0), (int)prv, 4);
            const double b = u - w * p + bias;
            double z = fast ? quotient(-b, w, rw) : -b / w;
            if (j == 0u) z = clamp0(z);
            const double lim = mu * from(z, 0), z2 = z * z;
            const double len2 = from(z2, 1) + from(z2, 2);
            if (beyond(len2, lim * lim)) {
                const double sc = slide_scale(lim, len2);
                if (j != 0u) z *= sc;
            }
            if (omega != 1.0) z = omega * z + (1.0 - omega) * p;
            d = z - p;
            if (moves) p = z;
        }
        if (!moves) d = 0.0;
        const double dn = from(d, 0), dt = from(d, 1), do_ = from(d, 2);
        const double P = dn * n_ + dt * t_ + do_ * o_, q = dt * o_ - do_ * t_;
        if (moves) {
            va += ima * P;
            wa -= ka * q;
            vb -= imb * P;
            wb -= kb * q;
        }
        r = d;
    }
    // r_j^2 on every lane
    __device__ __forceinline__ double residual() const
    {
        const double r1 = w * r, r2 = r1 * r1;
        return from(r2, 0) + from(r2, 1) + from(r2, 2);
    }
};

}  // namespace nbgs
