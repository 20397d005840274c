// flow.cu -- the NBGS solve as a dataflow over body versions.
//
// The sweeps relax the contacts colour by colour; the order that matters is
// only that every body sees its contacts in colour order.  So a contact does
// not wait for a colour to end anywhere: every body's velocity record carries
// a version, each contact waits until both of its bodies show the version its
// predecessor leaves, and stores the two records back with the next one.  The
// result is that of the sweeps in colour order, bit for bit.
//
// Versions.  A contact of colour c relaxed in pass k (pass 0 applies the
// initial impulses of a warm start, the sweeps follow) leaves (k << 9) | (c +
// 1) on its bodies, and ((k + 1) << 9) on a body whose last contact it is; it
// expects (k << 9) | (colour of the body's contact before it + 1), or (k <<
// 9) on a body whose first contact it is.  The 9-bit fields come from the
// bodies' colour masks (dep word in .w of the impulse, colour.cu).
//
// Memory.  The state and its version travel in one 128-bit word, loaded and
// stored as .b128 with relaxed gpu scope: such an access is single-copy
// atomic, so a word that shows the expected version holds that version's
// values, with no fence, flag or barrier.  A body takes two words in FP32
// (v, tag), (w, tag), and four in FP64 (each a double, half of a third one
// and the tag).  1/m and 1/I sit in a read-only array beside them.  In FP32 a
// pair of lanes moves the two halves of one body (a whole 32-byte sector per
// pair) and exchanges them by shuffles.
//
// Schedule.  A colour is cut into tiles of up to 32 contacts; the tiles of
// all colours, in colour order, are dealt to the warps in turn, the same in
// every pass, so that a contact's impulse stays with one lane.  A warp goes
// through its tiles in (pass, colour) order and a tile waits only for tiles
// that come earlier in that order, so with every warp resident (a cooperative
// launch) the earliest unfinished tile can always run.  Every wait is bounded.
#include <algorithm>
#include <mutex>
#include <vector>

#include "units.cuh"

namespace nbgs {

namespace {

template <class R> struct Mass2;
template <> struct Mass2<float> { using T = float2; };
template <> struct Mass2<double> { using T = double2; };

template <class R> struct FlowArgs {
    int64_t n;
    uint32_t nrec;                    // ids below it have a velocity record (n, or with subdomains every instance)
    uint4* tv;                        // versioned velocities, Words<R>::N per record
    const typename Mass2<R>::T* mass;  // (1/m, 1/I), kept for the way back
    const SweepRec<R>* rec;
    const SweepPre<R>* pre;
    R4<R>* p;                         // impulses and dep words, colour order
    const uint32_t* col_off;
    DevInfo* info;
    R mu, omega;
    double gdt_norm;
    int max_sweeps;
    double tol;
    int warm;
    int tile;                         // contacts per tile: a power of two, at most 32
    // subdomains: the bodies with several instances, whose extra ones follow
    // record n from ext_off on, and their velocities at the start of the sweep
    const uint32_t* shared;
    const uint32_t* ext_off;
    R4<R>* vacc;
    // batched scenes
    const uint32_t* scene_of;
    int64_t nscene;
    const R4<R>* scene_par;           // (mu, r^2 at the tolerance, r^2 at which R_k exceeds it, -) per scene
    const double* scene_vref;
    unsigned long long* scene_rk;     // 3 x nscene rotating slots of max r^2 (bits), then 3 of "some R above tol"
    uint32_t* scene_done;
    double* scene_res;
};

__device__ __forceinline__ unsigned long long bits_of(float x) { return __float_as_uint(x); }
__device__ __forceinline__ unsigned long long bits_of(double x) { return (unsigned long long)__double_as_longlong(x); }
__device__ __forceinline__ void from_bits(unsigned long long b, float& x) { x = __uint_as_float((uint32_t)b); }
__device__ __forceinline__ void from_bits(unsigned long long b, double& x) { x = __longlong_as_double((long long)b); }

__device__ __forceinline__ uint32_t body_a(const SweepRec<float>& r) { return __float_as_uint(r.a.x); }
__device__ __forceinline__ uint32_t body_a(const SweepRec<double>& r) { return (uint32_t)__double2loint(r.ids_bias.x); }

// R_k of a scene from the largest r^2 of its contacts
template <class R> __device__ __forceinline__ double scene_residual(R r2, double vref) { return (double)sqrt(r2) / vref; }

// The largest r^2 >= 0 whose residual (rounded to R first if asked: what the
// record of R_k holds) is at or below tol.  Non-negative numbers order like
// their bits and the residual does not fall as r^2 grows, so a bisection
// finds it; it starts next to (tol v_ref)^2.
template <class R> __device__ R r2_at_tol(double vref, double tol, bool rounded)
{
    auto meets = [&](unsigned long long b) {
        R x;
        from_bits(b, x);
        const double r = scene_residual<R>(x, vref);
        return (rounded ? (double)(R)r : r) <= tol;
    };
    const R t = (R)(tol * vref), guess = t * t;
    unsigned long long lo = 0ull, hi = bits_of(sizeof(R) == 4 ? (R)__int_as_float(0x7F800000) : (R)__longlong_as_double(0x7FF0000000000000LL));
    if (meets(hi)) lo = hi;   // an infinite tolerance
    const unsigned long long g = bits_of(guess);
    if (g > 32ull && g < hi && meets(g - 32ull)) lo = g - 32ull;
    if (g + 32ull < hi && !meets(g + 32ull)) hi = g + 32ull;
    while (hi - lo > 1ull) {   // meets(lo) and not meets(hi)
        const unsigned long long m = lo + (hi - lo) / 2ull;
        if (meets(m)) lo = m;
        else hi = m;
    }
    R x;
    from_bits(lo, x);
    return x;
}

// max r^2 of the scenes of a tile's live contacts: the contacts of a tile are
// mostly of one scene, whose maximum is then one atomic nobody waits for.
__device__ __forceinline__ void scene_max(unsigned long long* rk, uint32_t scene, bool live, bool lead,
                                          unsigned long long bits)
{
    const uint32_t m = __ballot_sync(kFull, live);   // some lane is
    const int first = __ffs((int)m) - 1;
    const uint32_t scene0 = __shfl_sync(kFull, scene, first);   // by every lane, live or not
    if (__all_sync(kFull, !live || scene == scene0)) {
        if (!live) bits = 0ull;
        // non-negative numbers order like their bits, NaN above them
        const uint32_t hi = __reduce_max_sync(kFull, (uint32_t)(bits >> 32));
        const uint32_t lo = __reduce_max_sync(kFull, (uint32_t)(bits >> 32) == hi ? (uint32_t)bits : 0u);
        if ((int)(threadIdx.x & 31) == first) atomicMax(rk + scene, (unsigned long long)hi << 32 | lo);
    } else if (live && lead) {
        atomicMax(rk + scene, bits);
    }
}

// What the sweeps start from.  The sweep count is theirs to write, but where
// there is no contact a kernel with votes by warps has nobody to do it.
// Contacts that found no colour of their own (kErrColours) share the last one:
// no order of versions holds for them, and the solve is an error already, so
// nothing is relaxed.  (Both here: in k_solve_flow they cost box-sized scenes 1 %.)
__device__ __forceinline__ void flow_begin(DevInfo* info, int max_sweeps)
{
    if (blockIdx.x != 0 || threadIdx.x != 0) return;
    info->sweeps_done = (uint32_t)max_sweeps;
    if ((info->err & kErrColours) != 0u) info->n_colours = info->n_shared = 0u;
}

// A body that takes impulses but has no contact: nobody reads or writes a
// versioned record of it (adj_off: null when there is no contact at all).  In a
// gas those are nearly all: 16M bodies with 34k contacts, solve of 10 sweeps 343
// us before there were versions, 413 with a copy of every body, 361 without
// theirs.  In a pile nearly every body has contacts and asking costs more than
// it spares (1M bodies, 3 sweeps, 359 -> 369 us): only scenes with at least eight
// bodies to a contact ask (finite is null otherwise).
__device__ __forceinline__ bool untouched(int64_t i, const uint8_t* finite, const uint32_t* adj_off)
{
    return finite != nullptr && finite[i] != 0 && (adj_off == nullptr || adj_off[i] == adj_off[i + 1]);
}

// Gravity, versions 0 and the mass array; of batched scenes (nscene > 0) also
// what their contacts ask for.  Bodies that nothing touches are done with.
template <class R>
__global__ void k_flow_init(int64_t n, R4<R>* vel, R gx, R gy, R gz, const uint8_t* __restrict__ finite,
                            const uint32_t* __restrict__ adj_off, uint4* __restrict__ tv,
                            typename Mass2<R>::T* __restrict__ mass, int64_t nscene, const double* __restrict__ mu,
                            const double* __restrict__ vref, double tol, R4<R>* __restrict__ par, DevInfo* info,
                            int max_sweeps)
{
    flow_begin(info, max_sweeps);
    for (int64_t sc = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; sc < nscene; sc += (int64_t)gridDim.x * blockDim.x) {
        R4<R> q;
        q.x = (R)mu[sc];
        q.y = r2_at_tol<R>(vref[sc], tol, false);
        q.z = r2_at_tol<R>(vref[sc], tol, true);
        q.w = R(0);
        par[sc] = q;
    }
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        R4<R> v, w;
        ld_body(vel + 2 * i, v, w);
        if (v.w > R(0)) {
            v.x += gx;
            v.y += gy;
            v.z += gz;
        }
        if (untouched(i, finite, adj_off)) {
            st_body(vel + 2 * i, v, w);
            continue;
        }
        typename Mass2<R>::T m;
        m.x = v.w;
        m.y = w.w;
        mass[i] = m;
        pack_body(tv + Words<R>::N * i, 0u, v, w);
    }
}

// The same with subdomains, whose versioned records take the place of the
// bodies' (tv is vel: a thread reads its record before it overwrites it) and
// of the instances after them.
template <class R>
__global__ void k_flow_init_sub(FlowArgs<R> A, R4<R>* vel, R gx, R gy, R gz, typename Mass2<R>::T* __restrict__ mass)
{
    flow_begin(A.info, A.max_sweeps);
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < A.n; i += (int64_t)gridDim.x * blockDim.x) {
        R4<R> v = vel[2 * i], w = vel[2 * i + 1];
        typename Mass2<R>::T m;
        m.x = v.w;
        m.y = w.w;
        mass[i] = m;
        if (v.w > R(0)) {
            v.x += gx;
            v.y += gy;
            v.z += gz;
        }
        pack_body(A.tv + Words<R>::N * i, 0u, v, w);
        const uint32_t e0 = A.ext_off[i], e1 = A.ext_off[i + 1];
        if (e0 == e1) continue;
        A.vacc[2 * i] = v;
        A.vacc[2 * i + 1] = w;
        for (uint32_t e = e0; e < e1; ++e) pack_body(A.tv + Words<R>::N * (A.n + e), 0u, v, w);
    }
}

// End of a pass for up to 32 bodies with several instances, a lane each: v <-
// v_acc + sum_p (instance_p - v_acc) over the instances in increasing
// subdomain (the body's own record first) once each has had its last contact
// of the pass (tag base | kDone); then every instance and v_acc restart from v
// in the next pass.  False when a wait gave up.  (Two instances asked for at a
// time polled the lines that the contacts write to: 3.78 ms instead of 3.20 for
// 50 sweeps of 1.57M contacts, a fifth of the 262k bodies shared; 3.99 with the
// sums as a phase of blocks that wait for their neighbours.)
constexpr uint32_t kDone = 511u;

template <class R>
__device__ __forceinline__ bool reduce_tile(const FlowArgs<R>& A, uint32_t q, uint32_t n_shared, uint32_t base)
{
    constexpr int N = Words<R>::N;
    const uint32_t t = 32u * q + (threadIdx.x & 31u);
    bool ok = true;
    if (t < n_shared) {
        const uint32_t i = A.shared[t], e0 = A.ext_off[i], cnt = A.ext_off[i + 1] - e0;
        const R4<R> v0 = A.vacc[2 * (int64_t)i], w0 = A.vacc[2 * (int64_t)i + 1];
        R4<R> av = v0, aw = w0;
        const long long t0 = clock64();
        for (uint32_t e = 0; e <= cnt && ok; ++e) {
            const uint4* rec = A.tv + N * (e == 0 ? (int64_t)i : A.n + e0 + e - 1);
            R4<R> v, w;
            for (int polls = 1;; ++polls) {
                uint32_t tags[4];
                load_body(rec, v, w, tags);
                bool there = true;
#pragma unroll
                for (int k = 0; k < N; ++k) there = there && tags[k] == (base | kDone);
                if (there) break;
                if ((polls & 255) == 0) {   // bounded like every other wait
                    if (clock64() - t0 > (1LL << 31)) atomicOr(&A.info->err, kErrTimeout);
                    if ((((volatile uint32_t*)&A.info->err)[0] & kErrTimeout) != 0u) {
                        ok = false;
                        break;
                    }
                }
            }
            av.x += v.x - v0.x;
            av.y += v.y - v0.y;
            av.z += v.z - v0.z;
            aw.x += w.x - w0.x;
            aw.y += w.y - w0.y;
            aw.z += w.z - w0.z;
        }
        if (ok) {
            A.vacc[2 * (int64_t)i] = av;
            A.vacc[2 * (int64_t)i + 1] = aw;
            for (uint32_t e = 0; e <= cnt; ++e)
                pack_body(A.tv + N * (e == 0 ? (int64_t)i : A.n + e0 + e - 1), base + 512u, av, aw);
        }
    }
    return __all_sync(kFull, ok) != 0;
}

// The solved velocities back into the body records (with subdomains in place),
// and the solve's outcome.
template <class R, bool Batch>
__global__ void k_flow_out(FlowArgs<R> A, R4<R>* vel, const uint8_t* __restrict__ finite,
                           const uint32_t* __restrict__ adj_off)
{
    const int64_t gtid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, gstride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i = gtid; i < A.n; i += gstride) {
        if (untouched(i, finite, adj_off)) continue;
        R4<R> v, w;
        uint32_t tags[4];
        load_body(A.tv + Words<R>::N * i, v, w, tags);
        const typename Mass2<R>::T m = A.mass[i];
        v.w = m.x;
        w.w = m.y;
        st_body(vel + 2 * i, v, w);
    }
    const int k = (int)A.info->sweeps_done;
    if (Batch) {   // scenes still short of their tolerance ran every sweep
        for (int64_t sc = gtid; sc < A.nscene; sc += gstride) {
            if (A.scene_done[sc] == 0) {
                R r2 = R(0);
                if (k > 0) from_bits(A.scene_rk[scene_slot(k - 1) * A.nscene + sc], r2);
                A.scene_done[sc] = (uint32_t)k;
                A.scene_res[sc] = scene_residual<R>(r2, A.scene_vref[sc]);
            }
        }
    }
    if (gtid == 0) {
        const double vref = v_ref_of(A.info, A.gdt_norm);
        A.info->residual =
            k > 0 ? __longlong_as_double((long long)A.info->rk_bits[rk_slot(k - 1)]) / (Batch ? 1.0 : vref) : 0.0;
        A.info->v_ref = vref;
    }
}

// Threads of a block and blocks per SM the kernels are compiled for.
template <class R, int L> struct FlowShape {
    static constexpr int threads = 256, blocks = sizeof(R) == 4 ? 2 : 1;
};
template <> struct FlowShape<float, 1> {
    static constexpr int threads = 128, blocks = 6;
};

// Records R_k = x v_ref for a warp and votes on the tolerance: 1 go on, 0 every
// one of the n voters is below it, -1 a wait gave up.
__device__ __noinline__ int warp_vote(DevInfo* info, int k, double x, bool below, uint32_t n)
{
    if (!(x <= 1e300)) x = __longlong_as_double(0x7FF0000000000000LL);
    atomicMax(&info->rk_bits[rk_slot(k)], (unsigned long long)__double_as_longlong(x));
    volatile uint32_t* flag = info->votes + 2 * k;
    if (!below) {
        flag[0] = 1u;
        return 1;
    }
    atomicAdd(info->votes + 2 * k + 1, 1u);
    const long long t0 = clock64();
    for (;;) {
        if (flag[0] != 0u) return 1;
        if (flag[1] == n) return 0;
        if ((((volatile uint32_t*)&info->err)[0] & kErrTimeout) || clock64() - t0 > (1LL << 31)) {
            atomicOr(&info->err, kErrTimeout);
            return -1;
        }
    }
}

// Vote: the tolerance test without a block waiting for its warps.  A warp with
// a contact above the tolerance says so at once, one without waits at the end
// of its sweep until another has or all are done.
template <class R, int L, bool Batch, bool Sub = false, bool Vote = false>
__global__ void __launch_bounds__((FlowShape<R, L>::threads), (FlowShape<R, L>::blocks)) k_solve_flow(FlowArgs<R> A)
{
    __shared__ uint32_t s_tile[kMaxColours + 1];   // first tile of every colour
    __shared__ uint32_t s_off[kMaxColours + 1];
    __shared__ int s_vote;
    const int ncol = min((int)A.info->n_colours, kMaxColours);
    const unsigned nb = gridDim.x;
    const int lane = threadIdx.x & 31;
    const uint32_t tw = (uint32_t)A.tile;
    tile_offsets(A.col_off, ncol, tw, s_off, s_tile);
    const uint32_t ntile = s_tile[ncol];
    // Warp w0 of the grid.  FP32, every warp with tiles: the warps of a block take
    // consecutive ones, whose bodies and records share lines.  Few tiles spread
    // over the SMs, warps 0 of all blocks first; so do FP64 ones, whose
    // arithmetic would pile up on the SMs a chain of contacts passes.  Sweeps,
    // ms, spread -> consecutive: FP32 8k 1.52 -> 1.36, 60k 2.05 -> 1.79, 250k
    // 1.52 -> 1.38, 500k 5.18 -> 4.94, 1M 8.43 -> 8.37, numbered z first 18.1 ->
    // 17.0; FP64 12k 1.07 -> 1.40, 40k 1.66 -> 1.90, 120k 3.16 -> 3.19.
    const uint32_t W = nb * (blockDim.x >> 5);
    const bool near_by = sizeof(R) == 4 && ntile > W;
    const uint32_t w0 = near_by ? blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)
                                : (threadIdx.x >> 5) * nb + blockIdx.x;
    // with subdomains the tiles of the shared bodies' sums follow the contacts'
    const uint32_t n_shared = Sub ? A.info->n_shared : 0u, ntot = ntile + (Sub ? (n_shared + 31u) / 32u : 0u);
    const bool work = w0 < ntot;
    const double vref = v_ref_of(A.info, A.gdt_norm);
    const int warm = A.warm ? 1 : 0;
    const int npass = A.max_sweeps + warm;
    bool ok = true;

    // lanes 2i and 2i + 1 of a lane per FP32 contact take contacts i and i +
    // 16 of a tile of 32: each access of a pair of lanes then covers
    // consecutive contacts, whose bodies tend to share lines
    const uint32_t unit = sizeof(R) == 4 && L == 1 ? (uint32_t)(lane >> 1) + 16u * (lane & 1) : (uint32_t)(lane / L);
    // a position in the tile order: tile T of colour c, the colour's tiles end
    // at tend; unit u's contact of it is slot base + T tw + u, if below send
    struct Pos {
        uint32_t T, tend, base, send;
        int c;
    };
    auto seek = [&](Pos& q, uint32_t T, int c) {
        while (T >= s_tile[c + 1]) ++c;
        q.T = T;
        q.c = c;
        q.tend = s_tile[c + 1];
        q.send = s_off[c + 1];
        q.base = s_off[c] - s_tile[c] * tw;
    };
    Unit<R, L> K;
    uint32_t s = 0;
    bool on = false;
    Pos at = {0u, 0u, 0u, 0u, 0};
    SweepRec<R> nrec;
    SweepPre<R> npre;
    R4<R> npp;
    auto read = [&](uint32_t sl) {
        nrec = ld_rec(A.rec + sl);
        npre = ld_pre(A.pre + sl);
        npp = A.p[sl];
    };
    // of a batch: the contact's scene and what that asks of a contact
    uint32_t na = 0, nscene = 0, scene = 0;
    R4<R> par = {};
    R prev = R(0);
    // the records of the warp's next tile: into registers, or, in the variant
    // whose many warps leave none to spare, into L1 (loads nobody waits for)
    constexpr bool Touch = sizeof(R) == 4 && L == 1;
    auto fetch = [&](const Pos& q, uint32_t& sl, bool& live) {
        sl = q.base + q.T * tw + unit;
        live = unit < tw && sl < q.send;
        if (!live) return;
        if constexpr (Touch) {
            uint32_t x;
            asm volatile("ld.global.b32 %0, [%1];" : "=r"(x) : "l"(A.rec + sl));
            if (Batch) na = x;   // the record's first word
            asm volatile("ld.global.b32 %0, [%1];" : "=r"(x) : "l"(A.pre + sl));
            asm volatile("ld.global.b32 %0, [%1];" : "=r"(x) : "l"(A.p + sl));
        } else {
            read(sl);
            if (Batch) na = body_a(nrec);
        }
    };
    auto scene_of = [&](bool live) { nscene = live ? A.scene_of[na] : 0u; };
    // prev: the scene's largest r^2 of the sweep before, complete since the barrier (NaN: no sweep yet)
    auto ask = [&](int sweep) {
        par = A.scene_par[scene];
        from_bits(sweep > 0 ? ((volatile unsigned long long*)A.scene_rk)[scene_slot(sweep - 1) * A.nscene + scene]
                            : ~0ull, prev);
    };
    // the contact fetched (slot s) becomes the unit's current one
    auto take = [&]() {
        if (on) {
            if (Touch) read(s);
            K.take(nrec, npre, npp, A.nrec);
        }
        // idle units read along with the first one, which every tile has
        const uint32_t q0 = __shfl_sync(kFull, K.qa, 0);
        if (!on) K.idle(q0);
    };
    if (work && (!Sub || w0 < ntile)) {
        seek(at, w0, 0);
        fetch(at, s, on);
        if (Batch) scene_of(on);
        take();
        scene = nscene;
    }
    if (Sub) at.T = w0;
    if (Vote && !work) return;
    // the tolerance as a residual in R, and where the FP64 division is not needed to tell
    const R near = Vote ? (R)(A.tol * vref) : R(0), slack = sizeof(R) == 4 ? R(1e-5) : R(1e-12);
    const bool clear = near > R(1e-15) && near < R(1e15);
    const R far2 = near * near * (R(1) + R(4) * slack);
    int k = 0;
    for (int pass = 0; pass < npass; ++pass) {
        const bool apply = pass < warm;
        k = pass - warm;
        if (!apply) {
            if (blockIdx.x == 0 && threadIdx.x == 0 && k + 1 >= kHistKept) A.info->rk_bits[rk_slot(k + 1)] = 0ull;
            if (Batch) {   // the slots of sweep k + 1 are neither read nor written during sweep k
                if (blockIdx.x == 0 && threadIdx.x == 0) A.scene_rk[3 * A.nscene + scene_slot(k + 1)] = 0ull;
                for (int64_t sc = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; sc < A.nscene;
                     sc += (int64_t)gridDim.x * blockDim.x)
                    A.scene_rk[scene_slot(k + 1) * A.nscene + sc] = 0ull;
            }
        }
        R rmax = R(0);
        bool over = false;   // a scene's contact above its tolerance
        bool said = false;   // this warp's is known to the others
        if (Batch) ask(apply ? 0 : k);
        const uint32_t base = (uint32_t)pass << 9;
        for (bool more = work; more && ok;) {
            if (Sub && at.T >= ntile) {   // a tile of sums
                ok = reduce_tile<R>(A, at.T - ntile, n_shared, base);
                if (!ok) break;
                more = at.T + W < ntot;
                const uint32_t Tn = more ? at.T + W : w0;
                if (Tn < ntile) {
                    seek(at, Tn, 0);
                    fetch(at, s, on);
                    take();
                }
                at.T = Tn;
                continue;
            }
            K.load(A.tv);
            // while the bodies' words are on their way: the warp's next tile
            // (the first one again at the end of a pass), whose records
            // depend on no other warp
            const bool wrap = at.T + W >= ntot;
            const uint32_t Tn = wrap ? w0 : at.T + W;
            const bool same = Tn == at.T;
            uint32_t sn = s;
            bool non = on;
            const uint32_t c1 = (uint32_t)at.c + 1u;
            if (!same && !(Sub && Tn >= ntile)) {
                if (wrap || Tn >= at.tend) seek(at, Tn, wrap ? 0 : at.c);
                at.T = Tn;
                fetch(at, sn, non);
            }
            if (Sub && Tn >= ntile) at.T = Tn;
            const uint32_t dep = on ? dep_bits(K.pp.w) : 0u;
            // a scene that met its tolerance in an earlier sweep is done
            const bool live = on && !(Batch && prev <= par.y);
            const R mu = Batch ? par.x : A.mu;
            const bool va = live && (dep & kDepListA) != 0u, vb = live && K.hasb && (dep & kDepListB) != 0u;
            const uint32_t ma = va ? ~0u : 0u, mb = vb ? ~0u : 0u;
            const uint32_t ea = base | (dep & 0x1FFu), eb = base | ((dep >> 11) & 0x1FFu);
            const uint32_t after = base | c1, next = base + 512u;
            // a shared body's instances go through its sum before the next pass
            const uint32_t enda = Sub && (dep & kDepSharedA) ? base | kDone : next;
            const uint32_t endb = Sub && (dep & kDepSharedB) ? base | kDone : next;
            const uint32_t oa = (dep & kDepLastA) ? enda : after, ob = (dep & kDepLastB) ? endb : after;
            if (!__all_sync(kFull, K.ready(ma, mb, ea, eb))) {
                const long long t0 = clock64();
                int polls = 0;
                for (;;) {
                    K.load(A.tv);
                    if (__all_sync(kFull, K.ready(ma, mb, ea, eb))) break;
                    if ((++polls & 255) == 0) {   // bounded like every other wait
                        bool give_up = (((volatile uint32_t*)&A.info->err)[0] & kErrTimeout) != 0u;
                        if (clock64() - t0 > (1LL << 31)) {
                            if (lane == 0) atomicOr(&A.info->err, kErrTimeout);
                            give_up = true;
                        }
                        if (__any_sync(kFull, give_up)) {
                            ok = false;
                            break;
                        }
                    }
                }
                if (!ok) break;
            }
            if (Batch && !same) scene_of(non);   // the next tile's: its record has arrived
            if (Batch && !__any_sync(kFull, live)) {
                // nothing to do in this tile
            } else if (apply) {
                K.template relax<true>(live, mu, A.omega);
                K.store(A.tv, va, vb, oa, ob);
            } else {
                K.template relax<false>(live, mu, A.omega);
                K.store(A.tv, va, vb, oa, ob);
                if (live) K.save(A.p + s);
                const R r2 = K.residual();
                if (Batch) {
                    over = over || (live && !(r2 <= par.z));
                    scene_max(A.scene_rk + scene_slot(k) * A.nscene, scene, live, lane % L == 0, bits_of(r2));
                } else {
                    rmax = live && above(r2, rmax) ? r2 : rmax;
                    if (Vote && !said && clear && __any_sync(kFull, rmax > far2)) {
                        said = true;
                        if (lane == 0) ((volatile uint32_t*)A.info->votes)[2 * k] = 1u;
                    }
                }
            }
            __syncwarp();   // the lanes of a unit read back what one of them saved
            more = !wrap;
            if (!same && (!Sub || Tn < ntile)) {
                s = sn;
                on = non;
                take();
                if (Batch) {
                    scene = nscene;
                    ask(apply ? 0 : k);
                }
            }
        }
        if (apply) continue;
        if (!Batch) rmax = sqrt(rmax);
        if (Vote) {
            if (!ok) break;
            for (int o = 16; o > 0; o >>= 1) rmax = fmax(rmax, __shfl_xor_sync(kFull, rmax, o));
            const double x = (double)rmax;
            bool below = false;
            if (!said && !(clear && rmax > near * (R(1) + slack)))
                below = (clear && rmax < near * (R(1) - slack)) || x / vref <= A.tol;
            const int v = lane == 0 ? warp_vote(A.info, k, x, below, min(W, ntot)) : 0;
            const int all = __shfl_sync(kFull, v, 0);
            if (all < 0) ok = false;
            if (all <= 0) break;
            continue;
        }
        // R_k is recorded by every warp; a test of it needs the whole block, and
        // every block near the rotating residual slots or for batched scenes
        const bool vote = !Batch && ncol > 0 && A.tol > 0.0 && k + 2 < kHistKept;
        const bool sync = ncol > 0 && !vote && (A.tol > 0.0 || Batch || k + 2 >= kHistKept);
        if (!vote && !sync) {
            if (!ok) break;
            if (work) {
                for (int o = 16; o > 0; o >>= 1) rmax = fmax(rmax, __shfl_xor_sync(0xffffffffu, rmax, o));
                if (lane == 0) {
                    double x = (double)rmax;
                    if (!(x <= 1e300)) x = __longlong_as_double(0x7FF0000000000000LL);
                    atomicMax(&A.info->rk_bits[rk_slot(k)], (unsigned long long)__double_as_longlong(x));
                }
            }
            continue;
        }
        if (!__syncthreads_and(ok)) {
            ok = false;
            break;
        }
        if (Batch) {
            if (__syncthreads_or(over) && threadIdx.x == 0) atomicMax(A.scene_rk + 3 * A.nscene + scene_slot(k), 1ull);
            if (!grid_barrier(A.info, nb)) {
                ok = false;
                break;
            }
            // the largest R_k and the scenes that met their tolerance in this
            // sweep, by the last warps of the grid: they have the fewest tiles
            for (int64_t sc = (int64_t)nb * blockDim.x - 1 - (blockIdx.x * (int64_t)blockDim.x + threadIdx.x);
                 sc < A.nscene; sc += (int64_t)nb * blockDim.x) {
                R r2;
                from_bits(((volatile unsigned long long*)A.scene_rk)[scene_slot(k) * A.nscene + sc], r2);
                if (r2 == R(0) && A.scene_done[sc] != 0) continue;
                const double rs = scene_residual<R>(r2, A.scene_vref[sc]);
                double x = (double)(R)rs;
                if (!(x <= 1e300)) x = __longlong_as_double(0x7FF0000000000000LL);
                atomicMax(&A.info->rk_bits[rk_slot(k)], (unsigned long long)__double_as_longlong(x));
                if (A.tol > 0.0 && A.scene_done[sc] == 0 && rs <= A.tol) {
                    A.scene_done[sc] = (uint32_t)(k + 1);
                    A.scene_res[sc] = rs;
                }
            }
            if (A.tol > 0.0 && ((volatile unsigned long long*)A.scene_rk)[3 * A.nscene + scene_slot(k)] == 0ull) break;
            continue;
        }
        const double rb = block_max_to<R>(rmax, &A.info->rk_bits[rk_slot(k)]);
        if (vote) {
            const int v = tol_vote(A.info, k, rb, vref, A.tol, nb, &s_vote);
            if (v < 0) ok = false;
            if (v <= 0) break;
            continue;
        }
        if (!grid_barrier(A.info, nb)) {
            ok = false;
            break;
        }
        const double Rk = __longlong_as_double((long long)((volatile unsigned long long*)A.info->rk_bits)[rk_slot(k)]) / vref;
        if (A.tol > 0.0 && Rk <= A.tol) break;
    }
    // sweeps run: k + 1 after a break at sweep k, and max_sweeps at the end
    if (blockIdx.x == 0 && threadIdx.x == 0 && ok)
        A.info->sweeps_done = (uint32_t)(A.max_sweeps == 0 ? 0 : min(k + 1, A.max_sweeps));
}

// Resident blocks per SM of a flow kernel at a block size, looked up once per device.
int flow_occ(int device, const void* fn, int threads)
{
    struct Known {
        int device, threads, blocks;
        const void* fn;
    };
    static std::mutex mu;
    static std::vector<Known> known;
    std::lock_guard<std::mutex> lock(mu);
    for (const Known& k : known)
        if (k.fn == fn && k.threads == threads && k.device == device) return k.blocks;
    int o = 0;
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&o, fn, threads, 0);
    cudaGetLastError();
    known.push_back({device, threads, o, fn});
    return o;
}

// Which kernel, and how many warps, for a scene of n bodies and C contacts.
//
// A pile has 2.7 contacts per body (6 at most) in 13 to 18 colours.  Up to
// some 10^5 contacts a sweep takes as long as its longest chain of contacts, so
// the contact itself has to be quick (more lanes) and a warp beyond the tiles
// of a colour only polls; above, it takes as long as the memory system needs
// for the contacts in flight, so they have to be many.  50 sweeps of a pile,
// ms, one GB300:
//   bodies                        30k    120k    250k    500k      1M
//   FP32, 2 lanes, 1 block/SM    0.86    1.21    2.06    4.95    9.70
//   FP32, 2 lanes, 2 blocks/SM   0.91    1.16    1.48    2.93    5.55
//   FP32, 1 lane,  6 blocks/SM   1.24    1.64    1.85    2.57    4.15
//   bodies                         1k     12k     30k     60k    120k
//   FP64, 4 lanes, 8 warps/SM    1.44    1.74    2.23    3.67    7.09
//   FP64, 1 lane,  4 warps/SM    3.14    4.20    4.43    4.43    5.31
//   FP64, 1 lane,  8 warps/SM    3.14    4.91    5.55    5.73    5.83
// (FP64 since the sliding scale is rsqrt(): 2 to 4 % less up to 30k, the same above.)
// The FP32 kernels give the same bits, so their line is drawn by what decides,
// the contacts (256 loose scenes, 1.1M bodies with 0.6M contacts, two steps:
// 17.1 ms with two lanes, 19.2 with one); the FP64 ones by the bodies, which
// do not change from step to step.
struct FlowPlan {
    const void* fn;
    int tile, warps, blocks_per_sm;   // contacts per tile, warps per block
};

template <class R, int L>
const void* flow_kernel(bool batch, bool sub)
{
    return sub     ? (const void*)k_solve_flow<R, L, false, true>
           : batch ? (const void*)k_solve_flow<R, L, true>
                   : (const void*)k_solve_flow<R, L, false>;
}

// A tolerance is voted on by warps (vote) where the chain of contacts bounds a
// sweep and by blocks where their number does: with the tolerance, ms,
//   bodies              1k FP64    2k     30k    250k   500k     1M
//   by blocks             1.55    6.81   1.90   2.00    5.18   8.40
//   by warps              1.42    6.00   1.77   2.19    6.74  10.03
template <class R>
FlowPlan flow_plan(int64_t n, int64_t C, bool batch, bool sub, bool vote)
{
    vote = vote && !batch && !sub;
    if (sizeof(R) == 4) {
        if (C < 245000)
            return {vote ? (const void*)k_solve_flow<float, 2, false, false, true> : flow_kernel<float, 2>(batch, sub),
                    16, 8, 1};
        if (C < 950000) return {flow_kernel<float, 2>(batch, sub), 16, 8, 2};
        return {flow_kernel<float, 1>(batch, sub), 32, 4, 6};
    }
    if (n < 64000)
        return {vote ? (const void*)k_solve_flow<double, 4, false, false, true> : flow_kernel<double, 4>(batch, sub),
                8, 8, 1};
    return {flow_kernel<double, 1>(batch, sub), 32, n < 250000 ? 4 : 8, 1};
}

}  // namespace

// The whole solve: gravity and versions, the passes, the body records.
template <class R>
nbgs_status run_flow(nbgs_scene* s, int max_sweeps, double tol, int warm)
{
    cudaStream_t st = s->stream;
    const int64_t n = s->n;
    FlowArgs<R> A;
    A.n = n;
    // the state-transfer staging buffer (13 doubles per body) holds the
    // versioned records and the masses during a solve; with subdomains the
    // velocity records, which have room for the instances, are versioned in
    // place.  Without contacts no instances are assigned (run_colour), and the
    // subdomain arrays hold an earlier step's or do not exist yet.
    const bool sub = s->prm.subdomain_mode != NBGS_SUB_NONE && !s->batch && s->n_contacts > 0;
    A.nrec = (uint32_t)(sub ? n + s->icap : n);
    A.tv = sub ? (uint4*)s->vel : (uint4*)s->stage;
    typename Mass2<R>::T* mass =
        (typename Mass2<R>::T*)((uint4*)s->stage + (size_t)Words<R>::N * std::max<int64_t>(n, 1));
    A.mass = mass;
    A.shared = s->shared;
    A.ext_off = s->ext_off;
    A.vacc = (R4<R>*)s->vacc;
    A.rec = (const SweepRec<R>*)s->srec;
    A.pre = (const SweepPre<R>*)s->spre;
    A.p = (R4<R>*)s->sp;
    A.col_off = s->col_off;
    A.info = s->info;
    A.mu = (R)s->prm.mu;
    A.omega = (R)s->prm.omega;
    const double* g = s->prm.gravity;
    A.gdt_norm = sqrt((g[0] * g[0] + g[1] * g[1]) + g[2] * g[2]) * s->prm.dt;
    A.max_sweeps = max_sweeps;
    A.tol = tol;
    A.warm = warm;
    A.scene_of = s->scene_of;
    A.nscene = s->batch ? s->n_scenes : 0;
    A.scene_par = (const R4<R>*)s->scene_par;
    A.scene_vref = s->scene_vref;
    A.scene_rk = s->scene_rk;
    A.scene_done = s->scene_done;
    A.scene_res = s->scene_res;
    // (near the rotating residual slots blocks meet at a barrier: they vote as blocks then)
    const bool vote = tol > 0.0 && max_sweeps + 2 < kHistKept && s->n_contacts > 0;
    const FlowPlan P = flow_plan<R>(s->n, known_contacts(s), s->batch, sub, vote);
    A.tile = P.tile;
    const void* fn = P.fn;
    const int threads = 32 * P.warps;
    int nblocks = std::min(flow_occ(s->device, fn, threads), P.blocks_per_sm) * s->num_sms;
    if (s->coop_blocks < s->max_coop_blocks) nblocks = std::min(nblocks, s->coop_blocks);   // set by nbgs_autotune
    if (nblocks < 1) return fail(s, NBGS_ECUDA, "solve: sweep kernel does not fit");
    const int T = 256, gb = grid_for(std::max<int64_t>(n, 1), T, 8, s->num_sms);
    const R gx = (R)(s->prm.dt * g[0]), gy = (R)(s->prm.dt * g[1]), gz = (R)(s->prm.dt * g[2]);
    // which bodies have contacts is known from this step's colouring
    const uint8_t* finite = !sub && 8 * known_contacts(s) <= n ? s->finite : nullptr;
    const uint32_t* lists = s->n_contacts > 0 ? s->adj_off : nullptr;
    if (sub)
        k_flow_init_sub<R><<<gb, T, 0, st>>>(A, (R4<R>*)s->vel, gx, gy, gz, mass);
    else
        k_flow_init<R><<<gb, T, 0, st>>>(n, (R4<R>*)s->vel, gx, gy, gz, finite, lists, A.tv, mass, A.nscene,
                                         s->scene_mu, s->scene_vref, tol, (R4<R>*)s->scene_par, s->info, max_sweeps);
    void* args[] = {&A};
    if (s->timing) cudaEventRecord(s->ev[8], st);
    const cudaError_t e = cudaLaunchCooperativeKernel(fn, dim3(nblocks), dim3(threads), args, 0, st);
    if (s->timing) {
        cudaEventRecord(s->ev[9], st);
        s->phase_launches[2] += 3;
        s->sweep_launches += 1;
    }
    if (e != cudaSuccess) return cuda_check(s, e, "solve: cooperative launch");
    if (s->batch) k_flow_out<R, true><<<gb, T, 0, st>>>(A, (R4<R>*)s->vel, finite, lists);
    else k_flow_out<R, false><<<gb, T, 0, st>>>(A, (R4<R>*)s->vel, finite, lists);
    return cuda_check(s, cudaGetLastError(), "solve");
}

template nbgs_status run_flow<float>(nbgs_scene*, int, double, int);
template nbgs_status run_flow<double>(nbgs_scene*, int, double, int);

}  // namespace nbgs
