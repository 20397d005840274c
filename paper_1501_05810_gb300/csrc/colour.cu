// colour.cu -- contact colouring and the colour-ordered sweep records.
//
// The subdomain numbers s_c(j) of Alg. 1 become colours: two contacts that
// share a body of finite mass never get the same colour, so all contacts of
// one colour can be relaxed at once with in-place velocity updates and no
// atomics, and the result equals the sequential NBGS in colour order.
//
//   k_colour_init   priority splitmix64(key ^ seed), body degrees
//   scan + k_adj_fill  body -> contact incidence lists (finite bodies only)
//   k_adj_sort_*    every incidence list in decreasing priority; each
//                   contact's successors in the lists of its bodies
//   k_colour_chase  first-fit greedy colouring in decreasing priority: a
//                   contact takes the smallest colour absent from the
//                   coloured prefixes of its bodies' lists as soon as all
//                   its predecessors have theirs
//   k_colour_hist, scan, k_colour_scatter
//                   stable counting sort by colour -> permutation
//   k_build_sweep   sweep records in colour order, initial impulses
#include <algorithm>

#include "relax.cuh"

namespace nbgs {

// Successor word of a contact in a body's list: the next contact (or
// kNoNext), and whether one comes before it.
constexpr uint32_t kNoNext = 0x7FFFFFFFu, kHasPrev = 1u << 31;

// Key of a contact in its own scene's numbering (bodies from 0, walls
// after the scene's bodies: shared planes, then the six box faces), so that
// batched scenes are coloured exactly as each would be alone.
__device__ __forceinline__ uint64_t local_key(uint32_t a, uint32_t b, const SceneView& V)
{
    if (!V.batch) return ((uint64_t)a << 32) | b;
    const uint32_t s = V.scene_of[a];
    const uint32_t off = V.scene_off[s], ns = V.scene_off[s + 1] - off;
    uint64_t lb;
    if (b < (uint64_t)V.n) {
        lb = b - off;
    } else {
        const uint64_t w = b - (uint64_t)V.n;
        lb = ns + (w < (uint64_t)V.nplanes ? w : V.nplanes + (w - V.nplanes - 6ull * s));
    }
    return ((uint64_t)(a - off) << 32) | lb;
}

// Priorities from the contacts' keys; body degrees from the incidence ends
// ib1, ib2 (the contact's bodies: the contact ends themselves for spheres,
// the members' bodies for composites; >= n marks a wall).
__global__ void k_colour_init(DCount Cc, int64_t n, const uint32_t* __restrict__ cj1, const uint32_t* __restrict__ cj2,
                              const uint32_t* __restrict__ ib1, const uint32_t* __restrict__ ib2,
                              const uint8_t* __restrict__ finite, uint64_t seed, SceneView V, uint32_t* __restrict__ deg,
                              uint64_t* __restrict__ prio, uint32_t* __restrict__ cstate, uint4* __restrict__ cpack,
                              unsigned long long* __restrict__ meet)
{
    const int64_t C = Cc.get();
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < C; c += (int64_t)gridDim.x * blockDim.x) {
        prio[c] = splitmix64(local_key(cj1[c], cj2[c], V) ^ seed);
        cstate[c] = kUncoloured;
        meet[c] = 0ull;
        const uint32_t a = ib1[c], b = ib2[c];
        const bool fa = finite[a] != 0, fb = b < n && finite[b];
        if (fa) atomicAdd(&deg[a], 1u);
        if (fb) atomicAdd(&deg[b], 1u);
        // the bodies whose incidence lists hold c (none: no list), successors later
        cpack[c] = make_uint4(fa ? a : kNoList, fb ? b : kNoList, kNoNext, kNoNext);
    }
}

__global__ void k_adj_fill(DCount Cc, int64_t n, const uint32_t* __restrict__ cj1, const uint32_t* __restrict__ cj2,
                           const uint8_t* __restrict__ finite, const uint32_t* __restrict__ adj_off,
                           uint32_t* __restrict__ fill, uint32_t* __restrict__ adj)
{
    const int64_t C = Cc.get();
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < C; c += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t a = cj1[c], b = cj2[c];
        if (finite[a]) adj[adj_off[a] + atomicAdd(&fill[a], 1u)] = (uint32_t)c;
        if (b < n && finite[b]) adj[adj_off[b] + atomicAdd(&fill[b], 1u)] = (uint32_t)c;
    }
}

// (prio, key) of d beats that of c: higher priority, ties to the lower key.
// Contacts are stored in canonical order, so the lower index is the lower key.
__device__ __forceinline__ bool beats(uint64_t pd, uint32_t d, uint64_t pc, uint32_t c)
{
    if (pd != pc) return pd > pc;
    return d < c;
}

// Colouring by priority-ordered incidence lists.  First-fit greedy
// colouring in decreasing priority gives each contact the smallest colour
// none of its predecessors (incident contacts that beat it) has.  With the
// incidence list of every body sorted by priority, the predecessors of c
// are the entries before c in the lists of its bodies.  A body's mask is the
// set of colours in the coloured prefix of its list; once the entries right
// before c in both lists are coloured, c's colour is the smallest one in
// neither mask.  Colouring c adds its colour to the masks and "arrives" at
// the next entry of either list; the last arrival at a contact (its only
// predecessor's, or the second of two) is followed by its colouring.  So the
// colours are those of the sequential greedy colouring whatever the order in
// which the threads come along, and no thread waits for another.

// Incidence lists in decreasing priority ("beats" order), kept as each
// contact's successors in the lists of its bodies (cpack z for its first
// body, w for its second).  Short lists (up to 16 contacts, every sphere
// scene) take a bitonic network in a thread's registers, of 8 entries where
// the lists of a warp allow it; longer ones a warp, lane l holding entries l,
// l + 32, ..., an entry's position being the number of entries that beat it,
// counted over the others broadcast by shuffles (one lane sorts lists beyond
// the warp's slots in place).
constexpr uint32_t kShortList = 16;
constexpr int kSortSlots = 8;   // entries per lane of the warp sort: lists of up to 256 contacts

__device__ __forceinline__ void set_next(uint4* cpack, uint32_t c, uint32_t x, uint32_t next, bool first)
{
    uint32_t* q = reinterpret_cast<uint32_t*>(cpack + c);
    q[q[0] == x ? 2 : 3] = next | (first ? 0u : kHasPrev);
}

// A list of m <= N entries at adj, sorted in registers.
template <uint32_t N>
__device__ __forceinline__ void sort_short(uint32_t x, uint32_t m, const uint32_t* __restrict__ adj,
                                           const uint64_t* __restrict__ prio, uint4* __restrict__ cpack)
{
    uint32_t id[N];
    uint64_t pr[N];
#pragma unroll
    for (uint32_t i = 0; i < N; ++i) id[i] = i < m ? adj[i] : 0xFFFFFFFFu;
#pragma unroll
    for (uint32_t i = 0; i < N; ++i) pr[i] = i < m ? prio[id[i]] : 0ull;   // padding sorts last
    // bitonic network: after it, entry i beats entry i + 1
#pragma unroll
    for (uint32_t k = 2; k <= N; k <<= 1) {
#pragma unroll
        for (uint32_t j = k >> 1; j > 0; j >>= 1) {
#pragma unroll
            for (uint32_t i = 0; i < N; ++i) {
                const uint32_t l = i ^ j;
                if (l <= i) continue;
                const bool first = (i & k) == 0;   // this half ends with i beating l
                const bool swap = first ? beats(pr[l], id[l], pr[i], id[i]) : beats(pr[i], id[i], pr[l], id[l]);
                if (swap) {
                    const uint32_t ti = id[i];
                    const uint64_t tp = pr[i];
                    id[i] = id[l];
                    pr[i] = pr[l];
                    id[l] = ti;
                    pr[l] = tp;
                }
            }
        }
    }
#pragma unroll
    for (uint32_t i = 0; i < N; ++i)
        if (i < m) set_next(cpack, id[i], x, i + 1 < m ? id[i + 1 < N ? i + 1 : i] : kNoNext, i == 0);
}

// Also empties the colour mask of every body with a list (the colouring
// reads no other body's) and collects the bodies with long lists.
__global__ void k_adj_sort_short(int64_t n, const uint8_t* __restrict__ finite, const uint32_t* __restrict__ adj_off,
                                 const uint32_t* __restrict__ adj, const uint64_t* __restrict__ prio,
                                 uint4* __restrict__ cpack, uint32_t* __restrict__ mask,
                                 uint32_t* __restrict__ longs, uint32_t* n_long)
{
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    // warp-uniform trip count: every lane takes part in the votes
    for (int64_t x0 = blockIdx.x * (int64_t)blockDim.x + (threadIdx.x & ~31u); x0 < n; x0 += stride) {
        const int64_t x = x0 + (threadIdx.x & 31u);
        uint32_t a0 = 0, m = 0;
        if (x < n && finite[x]) {
            a0 = adj_off[x];
            m = adj_off[x + 1] - a0;
        }
        if (m > 0) {
            uint4* mk = reinterpret_cast<uint4*>(mask + 8 * x);
            mk[0] = make_uint4(0u, 0u, 0u, 0u);
            mk[1] = make_uint4(0u, 0u, 0u, 0u);
        }
        if (m > kShortList) {
            longs[atomicAdd(n_long, 1u)] = (uint32_t)x;
            m = 0;
        }
        if (__any_sync(0xffffffffu, m > 8u)) sort_short<kShortList>((uint32_t)x, m, adj + a0, prio, cpack);
        else if (__any_sync(0xffffffffu, m > 0u)) sort_short<8>((uint32_t)x, m, adj + a0, prio, cpack);
    }
}

// One list of m entries (m <= 32 K) by the warp: lane l holds entries l,
// l + 32, ...; an entry's position is the number of entries that beat it.
template <int K>
__device__ __forceinline__ void warp_sort_list(uint32_t x, uint32_t a0, uint32_t m, uint32_t lane,
                                               uint32_t* adj, const uint64_t* __restrict__ prio,
                                               uint4* __restrict__ cpack)
{
    uint32_t id[K], rk[K];
    uint64_t pr[K];
#pragma unroll
    for (int k = 0; k < K; ++k) {
        const uint32_t i = lane + 32u * k;
        id[k] = i < m ? adj[a0 + i] : 0u;
        rk[k] = 0u;
    }
#pragma unroll
    for (int k = 0; k < K; ++k) pr[k] = lane + 32u * k < m ? prio[id[k]] : 0ull;
#pragma unroll
    for (int kc = 0; kc < K; ++kc) {
        if (32u * kc >= m) break;
        const uint32_t cnt = min(32u, m - 32u * kc);
        for (uint32_t l = 0; l < cnt; ++l) {
            const uint32_t idj = __shfl_sync(0xffffffffu, id[kc], l);
            const uint64_t prj = __shfl_sync(0xffffffffu, pr[kc], l);
#pragma unroll
            for (int k = 0; k < K; ++k)
                if (lane + 32u * k < m && beats(prj, idj, pr[k], id[k])) ++rk[k];
        }
    }
    __syncwarp();   // every entry read before any is overwritten
#pragma unroll
    for (int k = 0; k < K; ++k)
        if (lane + 32u * k < m) adj[a0 + rk[k]] = id[k];
    __syncwarp();
    for (uint32_t i = lane; i < m; i += 32u) set_next(cpack, adj[a0 + i], x, i + 1 < m ? adj[a0 + i + 1] : kNoNext, i == 0);
}

__global__ void k_adj_sort_long(const uint32_t* __restrict__ longs, const uint32_t* __restrict__ n_long,
                                const uint32_t* __restrict__ adj_off, uint32_t* __restrict__ adj,
                                const uint64_t* __restrict__ prio, uint4* __restrict__ cpack)
{
    const uint32_t lane = threadIdx.x & 31u;
    const int64_t nw = ((int64_t)gridDim.x * blockDim.x) >> 5, nl = *n_long;
    for (int64_t k = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5; k < nl; k += nw) {
        const uint32_t x = longs[k];   // the same for every lane of the warp
        const uint32_t a0 = adj_off[x], m = adj_off[x + 1] - a0;
        if (m <= 32u) warp_sort_list<1>(x, a0, m, lane, adj, prio, cpack);
        else if (m <= 64u) warp_sort_list<2>(x, a0, m, lane, adj, prio, cpack);
        else if (m <= 128u) warp_sort_list<4>(x, a0, m, lane, adj, prio, cpack);
        else if (m <= 32u * kSortSlots) warp_sort_list<kSortSlots>(x, a0, m, lane, adj, prio, cpack);
        else if (lane == 0) {   // beyond the slots: insertion sort by one lane
            for (uint32_t i = 1; i < m; ++i) {
                const uint32_t c = adj[a0 + i];
                const uint64_t pc = prio[c];
                uint32_t j = i;
                while (j > 0) {
                    const uint32_t d = adj[a0 + j - 1];
                    if (!beats(pc, c, prio[d], d)) break;
                    adj[a0 + j] = d;
                    --j;
                }
                adj[a0 + j] = c;
            }
            for (uint32_t q = 0; q < m; ++q)
                set_next(cpack, adj[a0 + q], x, q + 1 < m ? adj[a0 + q + 1] : kNoNext, q == 0);
        }
    }
}

// The colouring itself.  Each block works off a queue of its own in shared
// memory: contacts whose predecessors are all coloured, first its share of
// those that have none, then the ones its threads arrive at last.  In the
// order of the queue the fronts of all lists advance together, as in rounds
// over a global list, but without a barrier, a launch or a host in between:
// a link of a chain of contacts costs one pass of the block over its queue.
//
// A block that falls behind arrives last more often and so gets still more
// to do: one of 1064 ended up with 20 times its share of 2.75M contacts.  So a
// large scene is coloured in turns, launches that stop after some passes and
// leave their queues to a list that the next one deals out again; the last
// runs to the end.
//
// Where every list is short (up to 16 contacts: no colour above 30) an arrival
// brings the mask of its list along.  The first of two at a contact leaves it
// in the contact's word (31 colours and a mark for either list), the second
// finds it there in exchange: one compare-and-swap each, which is all that
// orders them; a pass is two memory latencies (the successors' words, the
// swaps).  Otherwise (Wide) the masks are kept in memory, 256 colours each,
// ordered by fences around a count of the arrivals.
// One kernel serves both, so that no launch is there for nothing.
//   us (ncu, cold)                            81k contacts   2.75M
//   rounds over a list, a launch per round        326         618
//   this, masks in memory and fences, one turn     98        1174
//   this, masks with the arrivals                  44         217
constexpr int kChaseThreads = 512;
constexpr uint32_t kChaseRing = 2048, kChaseRoom = 2 * kChaseThreads;   // a pass adds at most kChaseRoom

__device__ __forceinline__ void fence_gpu() { asm volatile("fence.acq_rel.gpu;" ::: "memory"); }

template <bool Wide>
__device__ __forceinline__ void chase(DCount Cc, const uint4* __restrict__ cpack, uint32_t* mask, uint32_t* cstate,
                                      unsigned long long* meet, const uint32_t* from, const uint32_t* from_count,
                                      uint32_t* to, uint32_t* to_count, int passes, DevInfo* info)
{
    extern __shared__ uint4 s_q[];                                         // kChaseRing contacts:
    uint32_t* const s_c = reinterpret_cast<uint32_t*>(s_q + kChaseRing);   // what they are, words and indices,
    uint2* const s_m = reinterpret_cast<uint2*>(s_c + kChaseRing);         // and the masks of their lists
    __shared__ uint32_t s_head, s_tail, s_spill;
    // what to start with: the contacts without predecessors, or those of a list
    const int64_t C = from ? (int64_t)*from_count : Cc.get(), stride = (int64_t)gridDim.x * kChaseThreads;
    const uint32_t tid = threadIdx.x;
    if (tid == 0) {
        s_head = s_tail = 0u;
        s_spill = kNoNext;
    }
    auto push = [&](uint32_t c, const uint4& q, uint32_t ma, uint32_t mb) {
        const uint32_t t = atomicAdd(&s_tail, 1u) % kChaseRing;
        s_c[t] = c;
        s_q[t] = q;
        if (!Wide) s_m[t] = make_uint2(ma, mb);
    };
    __syncthreads();
    // every branch on n is the same for the whole block
    for (int64_t seed = blockIdx.x * (int64_t)kChaseThreads;;) {
        uint32_t n = s_tail - s_head;
        __syncthreads();
        while (n < (uint32_t)kChaseThreads && seed < C) {
            const int64_t t = seed + tid;
            if (t < C && from) {
                const uint32_t c = from[t];
                const unsigned long long m = meet[c];
                push(c, cpack[c], (uint32_t)m, (uint32_t)(m >> 32));
            } else if (t < C) {
                const uint4 q = cpack[t];
                if (((q.z | q.w) & kHasPrev) == 0u) push((uint32_t)t, q, 0u, 0u);
            }
            seed += stride;
            __syncthreads();
            n = s_tail - s_head;
            __syncthreads();
        }
        if (n == 0u) {
            if (to_count) return;
            if (tid == 0) {
                uint32_t x = s_spill;
                for (int k = 0; k < kChaseThreads && x != kNoNext; ++k) {
                    const unsigned long long m = Wide ? 0ull : meet[x];
                    push(x, cpack[x], (uint32_t)m, (uint32_t)(m >> 32));
                    x = to[x];
                }
                s_spill = x;
            }
            __syncthreads();
            n = s_tail - s_head;
            __syncthreads();
            if (n == 0u) return;
        }
        // a queue that is full, or whose turn is over, gives its newest away;
        // their words are theirs alone by now
        const bool over = to_count && --passes < 0 && seed >= C;
        while (n > (over ? 0u : kChaseRing - kChaseRoom)) {
            const uint32_t k = min(n, (uint32_t)kChaseThreads), t = (s_tail - 1u - tid) % kChaseRing, c = s_c[t];
            if (tid < k && !Wide) meet[c] = (unsigned long long)s_m[t].y << 32 | s_m[t].x;
            if (to_count) {
                if (tid == 0) s_spill = atomicAdd(to_count, k);
                __syncthreads();
                if (tid < k) to[s_spill + tid] = c;
            } else if (tid < k) {   // the block's own, linked by contact
                to[c] = atomicExch(&s_spill, c);
            }
            __syncthreads();
            if (tid == 0) s_tail -= k;
            __syncthreads();
            n -= k;
        }
        if (over) return;
        const uint32_t take = min(n, (uint32_t)kChaseThreads);
        const uint32_t at = (s_head + tid) % kChaseRing;
        const uint32_t c = s_c[at];
        const uint4 q = s_q[at];
        uint2 m = make_uint2(0u, 0u);
        if (!Wide) m = s_m[at];
        __syncthreads();
        if (tid == 0) s_head += take;
        if (tid < take) {
            const uint32_t a = q.x, b = q.y, e0 = q.z & kNoNext, e1 = q.w & kNoNext;
            const bool fa = a != kNoList, fb = b != kNoList, n0 = e0 != kNoNext, n1 = e1 != kNoNext;
            const uint4 z = make_uint4(0u, 0u, 0u, 0u);
            const uint4 q0 = n0 ? cpack[e0] : z, q1 = n1 ? cpack[e1] : z;
            const bool two0 = (q0.z & q0.w & kHasPrev) != 0u, two1 = (q1.z & q1.w & kHasPrev) != 0u;
            if constexpr (!Wide) {
                const uint32_t col = (uint32_t)__ffs(~(m.x | m.y)) - 1u;   // at most 30: 15 predecessors in either list
                cstate[c] = col;
                m.x |= 1u << col;
                m.y |= 1u << col;
                // a list's last contact leaves the body's mask
                if (fa && !n0) mask[8 * (int64_t)a] = m.x;
                if (fb && !n1) mask[8 * (int64_t)b] = m.y;
                // which of a successor's lists this one is, and what was there
                const bool first0 = q0.x == a, first1 = q1.x == b;
                const unsigned long long w0 = (unsigned long long)(m.x | kHasPrev) << (first0 ? 0 : 32);
                const unsigned long long w1 = (unsigned long long)(m.y | kHasPrev) << (first1 ? 0 : 32);
                unsigned long long o0 = 0ull, o1 = 0ull;
                if (n0 && two0) o0 = atomicCAS(meet + e0, 0ull, w0);
                if (n1 && two1) o1 = atomicCAS(meet + e1, 0ull, w1);
                if (n0 && (!two0 || o0 != 0ull)) {
                    o0 |= w0;
                    push(e0, q0, (uint32_t)o0 & ~kHasPrev, (uint32_t)(o0 >> 32) & ~kHasPrev);
                }
                if (n1 && (!two1 || o1 != 0ull)) {
                    o1 |= w1;
                    push(e1, q1, (uint32_t)o1 & ~kHasPrev, (uint32_t)(o1 >> 32) & ~kHasPrev);
                }
            } else {
                const uint4* ma = reinterpret_cast<const uint4*>(mask + 8 * (int64_t)a);
                const uint4* mb = reinterpret_cast<const uint4*>(mask + 8 * (int64_t)b);
                const uint4 a_lo = fa ? __ldcg(ma) : z, a_hi = fa ? __ldcg(ma + 1) : z;
                const uint4 b_lo = fb ? __ldcg(mb) : z, b_hi = fb ? __ldcg(mb + 1) : z;
                const uint32_t wa[8] = {a_lo.x, a_lo.y, a_lo.z, a_lo.w, a_hi.x, a_hi.y, a_hi.z, a_hi.w};
                const uint32_t wb[8] = {b_lo.x, b_lo.y, b_lo.z, b_lo.w, b_hi.x, b_hi.y, b_hi.z, b_hi.w};
                uint32_t col = kMaxColours, va = 0u, vb = 0u;
#pragma unroll
                for (int k = 7; k >= 0; --k) {
                    const uint32_t free = ~(wa[k] | wb[k]);
                    if (free) {
                        col = 32u * k + (__ffs(free) - 1);
                        va = wa[k];
                        vb = wb[k];
                    }
                }
                if (col >= (uint32_t)kMaxColours) {
                    atomicOr(&info->err, kErrColours);
                    col = kMaxColours - 1;
                    va = wa[7];
                    vb = wb[7];
                }
                cstate[c] = col;
                const uint32_t bit = 1u << (col & 31u), wd = col >> 5;
                // only c, the front of a and of b, writes their masks
                if (fa) __stcg(mask + 8 * (int64_t)a + wd, va | bit);
                if (fb) __stcg(mask + 8 * (int64_t)b + wd, vb | bit);
                fence_gpu();   // the masks before the arrivals
                unsigned long long o0 = 0ull, o1 = 0ull;
                if (n0 && two0) o0 = atomicAdd(meet + e0, 1ull);
                if (n1 && two1) o1 = atomicAdd(meet + e1, 1ull);
                fence_gpu();   // the arrivals before the masks that their contacts read
                if (n0 && (!two0 || o0 != 0ull)) push(e0, q0, 0u, 0u);
                if (n1 && (!two1 || o1 != 0ull)) push(e1, q1, 0u, 0u);
            }
        }
        __syncthreads();
    }
}

__global__ void __launch_bounds__(kChaseThreads)
k_colour_chase(DCount Cc, const uint4* __restrict__ cpack, uint32_t* mask, uint32_t* cstate, unsigned long long* meet,
               const uint32_t* from, const uint32_t* from_count, uint32_t* to, uint32_t* to_count, int passes,
               DevInfo* info)
{
    if (info->n_long != 0u) chase<true>(Cc, cpack, mask, cstate, meet, from, from_count, to, to_count, passes, info);
    else chase<false>(Cc, cpack, mask, cstate, meet, from, from_count, to, to_count, passes, info);
}

// Stable counting sort of the contacts by colour, in tiles: contacts of a
// colour stay in canonical order.  The colours come straight from the
// colouring's states; the scatter also writes the inverse permutation, the
// colours' offsets and their number.
constexpr int kSortThreads = 256, kSortItems = 16, kSortTile = kSortThreads * kSortItems, kSortWarps = kSortThreads / 32;

__global__ void __launch_bounds__(kSortThreads)
k_colour_hist(DCount Cc, const uint32_t* __restrict__ cstate, uint32_t* __restrict__ hist, int64_t nblocks,
              DevInfo* info)
{
    __shared__ uint32_t h[kMaxColours];
    const int64_t C = Cc.get();
    h[threadIdx.x] = 0;
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * kSortTile;
#pragma unroll
    for (int k = 0; k < kSortItems; ++k) {
        const int64_t c = base + (int64_t)k * kSortThreads + threadIdx.x;
        if (c >= C) continue;
        uint32_t col = cstate[c];
        if (col >= (uint32_t)kMaxColours) {   // uncoloured: report, keep indices in bounds
            atomicOr(&info->err, kErrColours);
            col = kMaxColours - 1;
        }
        atomicAdd(&h[col], 1u);
    }
    __syncthreads();
    hist[(int64_t)threadIdx.x * nblocks + blockIdx.x] = h[threadIdx.x];
}

__global__ void __launch_bounds__(kSortThreads)
k_colour_scatter(DCount Cc, const uint32_t* __restrict__ cstate, const uint32_t* __restrict__ hist_scan,
                 int64_t nblocks, uint32_t* __restrict__ perm, uint32_t* __restrict__ inv,
                 uint32_t* __restrict__ col_off, DevInfo* info)
{
    const int64_t C = Cc.get();
    __shared__ uint32_t cnt[kSortWarps][kMaxColours];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
    const int d0 = threadIdx.x;   // a thread per colour
    static_assert(kSortThreads == kMaxColours, "a thread per colour");
#pragma unroll
    for (int ww = 0; ww < kSortWarps; ++ww) cnt[ww][d0] = 0;
    if (blockIdx.x == 0) {
        const uint32_t s = hist_scan[(int64_t)d0 * nblocks];
        const uint32_t e = d0 + 1 < kMaxColours ? hist_scan[(int64_t)(d0 + 1) * nblocks] : (uint32_t)C;
        col_off[d0] = s;
        if (d0 == 0) col_off[kMaxColours] = (uint32_t)C;
        if (e > s) atomicMax(&info->n_colours, (uint32_t)d0 + 1u);
    }
    const uint32_t goff = hist_scan[(int64_t)d0 * nblocks + blockIdx.x];
    __syncthreads();
    const uint32_t lt = (1u << lane) - 1u;
    const int64_t base = (int64_t)blockIdx.x * kSortTile + (int64_t)w * (kSortItems * 32);
    uint32_t key[kSortItems], rank[kSortItems];
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
        const int64_t c = base + r * 32 + lane;
        const bool valid = c < C;
        key[r] = valid ? min(cstate[c], (uint32_t)kMaxColours - 1u) : 0u;
        const uint32_t peers = __match_any_sync(0xffffffffu, valid ? key[r] : 0x100u);
        const uint32_t before = cnt[w][key[r]];
        __syncwarp();
        if (valid && (peers & lt) == 0) cnt[w][key[r]] = before + __popc(peers);
        __syncwarp();
        rank[r] = before + __popc(peers & lt);
    }
    __syncthreads();
    // the tile's slots of each colour, warp by warp (warp order = input order)
    uint32_t sum = goff;
#pragma unroll
    for (int ww = 0; ww < kSortWarps; ++ww) {
        const uint32_t t = cnt[ww][d0];
        cnt[ww][d0] = sum;
        sum += t;
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSortItems; ++r) {
        const int64_t c = base + r * 32 + lane;
        if (c < C) {
            const uint32_t pos = cnt[w][key[r]] + rank[r];
            perm[pos] = (uint32_t)c;
            inv[c] = pos;
        }
    }
}

// With subdomains: what the ends of a contact need to know of their instances.
struct SubView {
    const uint32_t* inst;      // two instances per contact (null: no subdomains)
    const uint32_t* ext_off;   // a body's extra instances
    const uint32_t* ends;      // two dependency ends per contact, of bodies with several instances
    int jacobi;                // an instance per contact, one colour
};

// Dependency ends (as dep_end) of the contacts of every body with several
// instances: a contact comes after those of the same instance and a lower
// colour.  A thread per body, which looks its list up once; for each contact
// to look through its bodies' lists instead cost 120 us with 1.57M contacts.
__global__ void k_sub_ends(const uint32_t* __restrict__ shared, const uint32_t* __restrict__ adj_off,
                           const uint32_t* __restrict__ adj, const uint32_t* __restrict__ inst,
                           const uint32_t* __restrict__ cj1, const uint32_t* __restrict__ cstate,
                           const DevInfo* __restrict__ info, uint32_t* __restrict__ ends)
{
    const int64_t ns = info->n_shared;
    for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < ns; t += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t x = shared[t], e0 = adj_off[x], m = adj_off[x + 1] - e0;
        constexpr uint32_t kKept = 16;   // entries kept at hand; longer lists read theirs again
        uint32_t slot[kKept], col[kKept];
        auto look = [&](uint32_t e, uint32_t& s, uint32_t& k) {
            const uint32_t d = adj[e0 + e];
            s = inst[2 * (int64_t)d + (cj1[d] == x ? 0 : 1)];
            k = cstate[d] & 0xFFu;
        };
        for (uint32_t e = 0; e < min(m, kKept); ++e) look(e, slot[e], col[e]);
        for (uint32_t e = 0; e < m; ++e) {
            uint32_t s, k, pred = 0u;
            bool last = true;
            if (e < kKept) {
                s = slot[e];
                k = col[e];
            } else {
                look(e, s, k);
            }
            for (uint32_t f = 0; f < m; ++f) {
                uint32_t sf, kf;
                if (f < kKept) {
                    sf = slot[f];
                    kf = col[f];
                } else {
                    look(f, sf, kf);
                }
                if (sf != s) continue;
                if (kf < k) pred = max(pred, kf + 1u);
                if (kf > k) last = false;
            }
            const uint32_t d = adj[e0 + e];
            ends[2 * (int64_t)d + (cj1[d] == x ? 0 : 1)] = pred | (last ? kDepLastA : 0u) | kDepListA;
        }
    }
}

// End `side` of contact c (colour col) at body x.
__device__ __forceinline__ uint32_t sub_end(const SubView& S, uint32_t x, int side, int64_t c, uint32_t col,
                                            const uint32_t* __restrict__ mask, bool& several)
{
    several = S.ext_off[x + 1] != S.ext_off[x];
    if (S.jacobi) return kDepLastA | kDepListA;
    return several ? S.ends[2 * c + side] : dep_end(mask + 8 * (int64_t)x, col);
}

// Sweep record inv[c] <- canonical contact c; initial impulse from the
// previous step (world frame, re-projected onto the new frame and the cone)
// or zero.  A thread per canonical contact: the contact arrays and the
// previous step's rows are read in order, the records written scattered.
template <class R>
__global__ void k_build_sweep(DCount Cc, int64_t n, const uint32_t* __restrict__ inv, const uint32_t* __restrict__ cj1,
                              const uint32_t* __restrict__ cj2, SubView S,
                              const double4_32a* __restrict__ cgeo,
                              const double2* __restrict__ clev, double dt, double beta, double mu_all, SceneView V,
                              int warm,
                              const uint32_t* __restrict__ prev_row_off, const uint32_t* __restrict__ prev_j2,
                              const double4_32a* __restrict__ prev_P, int64_t prev_cap,
                              const uint32_t* __restrict__ cstate, const uint4* __restrict__ cpack,
                              const uint32_t* __restrict__ mask, const R4<R>* __restrict__ vel,
                              SweepRec<R>* __restrict__ rec, R4<R>* __restrict__ p, SweepPre<R>* __restrict__ pre)
{
    const int64_t C = Cc.get();
    for (int64_t c = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; c < C; c += (int64_t)gridDim.x * blockDim.x) {
        const uint32_t s = inv[c];
        const uint32_t a = cj1[c], b = cj2[c];
        // the velocity records the sweep reads: the bodies, or with subdomains
        // their instances for the contact's subdomain
        const uint32_t ra = S.inst ? S.inst[2 * (int64_t)c] : a, rb = S.inst ? S.inst[2 * (int64_t)c + 1] : b;
        const double4_32a g = cgeo[c];
        const double2 l = clev[c];
        // eq. (nonpenetration): gap term xi/dt, scaled by beta when xi < 0
        const double xs = g.w >= 0.0 ? g.w : beta * g.w;
        const double bias = xs / dt;
        SweepRec<R> r;
        if constexpr (sizeof(R) == 4) {
            r.a = make_float4(__uint_as_float(ra), __uint_as_float(rb), (float)l.x, (float)l.y);
            r.b = make_float4((float)g.x, (float)g.y, (float)g.z, (float)bias);
        } else {
            r.ids_bias = make_double2(__longlong_as_double((long long)(((uint64_t)rb << 32) | ra)), bias);
            r.lev = make_double2(l.x, l.y);
            r.nxy = make_double2(g.x, g.y);
            // the factor of the tangent basis (tangent_basis)
            r.nz_ = make_double2(g.z, -1.0 / (copysign(1.0, g.z) + g.z));
        }
        rec[s] = r;
        {
            const bool dyn_b = b < (uint64_t)n;
            const R ima = vel[2 * (int64_t)a].w, iIa = vel[2 * (int64_t)a + 1].w;
            const R imb = dyn_b ? vel[2 * (int64_t)b].w : R(0), iIb = dyn_b ? vel[2 * (int64_t)b + 1].w : R(0);
            SweepPre<R> x;
            // the levers as the records hold them
            const R la = (R)l.x, lb = (R)l.y, nz = (R)g.z;
            const R wn = ima + imb, wt = wn + iIa * la * la + iIb * lb * lb;
            x.m.x = ima;
            x.m.y = imb;
            x.m.z = la * iIa;
            x.m.w = lb * iIb;
            if constexpr (sizeof(R) == 4) x.w = make_float4(wt, 1.f / wn, 1.f / wt, -1.f / (copysignf(1.f, nz) + nz));
            else x.w = make_double4_32a(wn, wt, 1.0 / wn, 1.0 / wt);
            pre[s] = x;
        }
        // the previous world impulse in the new contact frame, projected onto
        // the friction cone; in the sweep precision (FP64 arithmetic is scarce
        // on this GPU, and an FP32 sweep starts from an FP32 impulse anyway)
        R pn = R(0), pt = R(0), po = R(0);
        uint32_t dep = 0u;
        {
            const uint32_t col = cstate[c] & 0xFFu;
            const uint4 q = cpack[c];
            if (S.inst) {
                bool sa = false, sb = false;
                if (q.x != kNoList) dep |= sub_end(S, q.x, 0, c, col, mask, sa);
                if (q.y != kNoList) dep |= sub_end(S, q.y, 1, c, col, mask, sb) << 11;
                dep |= (sa ? kDepSharedA : 0u) | (sb ? kDepSharedB : 0u);
            } else {
                if (q.x != kNoList) dep |= dep_end(mask + 8 * (int64_t)q.x, col);
                if (q.y != kNoList) dep |= dep_end(mask + 8 * (int64_t)q.y, col) << 11;
            }
        }
        if (warm) {
            const uint32_t e = prev_row_off[a + 1];
            for (uint32_t t = prev_row_off[a]; t < e && t < prev_cap; ++t) {
                if (prev_j2[t] != b) continue;
                const double4_32a P = prev_P[t];
                const R mu = (R)(V.batch ? V.mu[V.scene_of[a]] : mu_all);
                const R nx = (R)g.x, ny = (R)g.y, nz = (R)g.z, Px = (R)P.x, Py = (R)P.y, Pz = (R)P.z;
                dep |= kDepFound;   // read by the network warm start
                R tx, ty, tz, ox, oy, oz;
                tangent_basis<R>(nx, ny, nz, tx, ty, tz, ox, oy, oz);
                pn = nx * Px + ny * Py + nz * Pz;
                if (!(pn > R(0))) pn = R(0);
                pt = tx * Px + ty * Py + tz * Pz;
                po = ox * Px + oy * Py + oz * Pz;
                const R lim = mu * pn, len = sqrt(pt * pt + po * po);
                if (len > lim) {
                    if (len > R(0)) {
                        pt *= lim / len;
                        po *= lim / len;
                    } else {
                        pt = po = R(0);
                    }
                }
                break;
            }
        }
        R4<R> q;
        q.x = pn;
        q.y = pt;
        q.z = po;
        dep_store(dep, q.w);
        p[s] = q;
    }
}

nbgs_status run_colour(nbgs_scene* s)
{
    if (!s->detected) return fail(s, NBGS_EINVAL, "colour_contacts: call detect_contacts first");
    cudaStream_t st = s->stream;
    // C: the count, or in device-sized steps the capacity the launches are
    // sized for (the kernels read the count, Cn, on the device)
    const int64_t C = s->n_contacts, n = s->n;
    const DCount Cn = contact_count(s);
    if (s->timing) cudaEventRecord(s->ev[2], st);
    cudaMemsetAsync(&s->info->n_colours, 0, sizeof(uint32_t), st);
    cudaMemsetAsync(&s->info->n_shared, 0, 2 * sizeof(uint32_t), st);   // no shared bodies until assigned
    const bool sub = s->prm.subdomain_mode != NBGS_SUB_NONE;
    const bool jacobi = s->prm.subdomain_mode == NBGS_SUB_JACOBI;
    if (C > 0) {
        const int T = 256;
        const int gb = grid_for(C, T, 8, s->num_sms);
        // the conflict graph: contacts sharing a body of finite mass (for
        // composites the body of a member, not the member)
        if (s->composite) {
            nbgs_status rc = run_comp_ends(s);
            if (rc != NBGS_OK) return rc;
        }
        const uint32_t* ib1 = s->composite ? s->cb1 : s->cj1;
        const uint32_t* ib2 = s->composite ? s->cb2 : s->cj2;
        const uint8_t* finc = s->composite ? s->bfinite : s->finite;
        const int64_t ninc = s->composite ? s->nb : n;
        cudaMemsetAsync(s->deg, 0, (ninc + 1) * sizeof(uint32_t), st);
        k_colour_init<<<gb, T, 0, st>>>(Cn, ninc, s->cj1, s->cj2, ib1, ib2, finc, s->prm.colour_seed, scene_view(s),
                                        s->deg, s->cprio, s->cstate, s->cpack, s->cmeet);
        nbgs_status rc = exclusive_scan_u32(s, s->deg, s->adj_off, ninc, nullptr);
        if (rc != NBGS_OK) return rc;
        cudaMemsetAsync(s->deg, 0, (ninc + 1) * sizeof(uint32_t), st);
        k_adj_fill<<<gb, T, 0, st>>>(Cn, ninc, ib1, ib2, finc, s->adj_off, s->deg, s->adj);
        if (sub) {
            rc = run_subdomains(s);
            if (rc != NBGS_OK) return rc;
        }
        s->sub_count = sub ? C : -1;
        if (jacobi) {
            // non-linear block Jacobi: no contact sees another's reaction of
            // the same sweep, so a single colour
            cudaMemsetAsync(s->cstate, 0, C * sizeof(uint32_t), st);
        } else {
            cudaMemsetAsync(&s->info->n_long, 0, sizeof(uint32_t), st);
            k_adj_sort_short<<<grid_for(ninc, T, 8, s->num_sms), T, 0, st>>>(ninc, finc, s->adj_off, s->adj, s->cprio,
                                                                              s->cpack, s->cmask, s->clist[0],
                                                                              &s->info->n_long);
            k_adj_sort_long<<<8 * s->num_sms, T, 0, st>>>(s->clist[0], &s->info->n_long, s->adj_off, s->adj, s->cprio,
                                                           s->cpack);
            // in turns of several passes where a block would fall far behind:
            // colouring phase, us, 18 colours     117k  474k  717k  1.01M  5.99M  18.0M contacts
            //   one turn                           171   229   280   610
            //   7 turns of 9 passes                238   303   340   397   1628   6902
            //   12 turns of 9 passes                                       1690   5775
            // (16 colours, 8.28M: 2345 with 7 turns, 2480 with 12; 18.0M by rounds of a
            // launch each 5745).  Lists beyond 16 contacts, 3.16M / 8.69M: one turn 1233 /
            // 5019, 7 turns 1048 / 3120; 1.96M of composites 1303 / 1338.
            const int64_t known = known_contacts(s);
            const int turns = known < 800000 ? 1 : known < 12000000 ? 7 : kChaseTurns, passes = 9;
            const int gc = grid_for(C, kChaseThreads, 3, s->num_sms);
            uint32_t* cnt = s->info->chase_count;
            cudaMemsetAsync(cnt, 0, kChaseTurns * sizeof(uint32_t), st);
            const size_t smem = kChaseRing * (sizeof(uint4) + sizeof(uint32_t) + sizeof(uint2));
            rc = cuda_check(s, cudaFuncSetAttribute((const void*)k_colour_chase, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                                    (int)smem), "colour: queues");
            for (int k = 0; k < turns && rc == NBGS_OK; ++k) {
                k_colour_chase<<<gc, kChaseThreads, smem, st>>>(
                    Cn, s->cpack, s->cmask, s->cstate, s->cmeet, k ? s->clist[(k + 1) & 1] : nullptr,
                    k ? cnt + k - 1 : nullptr, s->clist[k & 1], k + 1 < turns ? cnt + k : nullptr, passes, s->info);
                rc = cuda_check(s, cudaGetLastError(), "colour: turns");
            }
            if (rc != NBGS_OK) return rc;
            if (s->timing) s->phase_launches[1] += 2 + turns;
        }
        const int64_t nbs = (C + kSortTile - 1) / kSortTile;
        if (kMaxColours * nbs > s->sort_hist_len) return fail(s, NBGS_EINVAL, "colour: histogram buffer too small");
        k_colour_hist<<<(unsigned)nbs, kSortThreads, 0, st>>>(Cn, s->cstate, s->sort_hist, nbs, s->info);
        rc = exclusive_scan_u32(s, s->sort_hist, s->sort_hist, kMaxColours * nbs, nullptr);
        if (rc != NBGS_OK) return rc;
        k_colour_scatter<<<(unsigned)nbs, kSortThreads, 0, st>>>(Cn, s->cstate, s->sort_hist, nbs, s->perm, s->inv,
                                                                 s->col_off, s->info);
        const int warm = (s->prm.warm_start != NBGS_WARM_NONE && s->have_prev) ? 1 : 0;
        uint32_t* ends = (uint32_t*)s->cprio;   // the priorities have served
        const SubView S{sub ? s->inst : nullptr, s->ext_off, ends, jacobi ? 1 : 0};
        if (sub && !jacobi)
            k_sub_ends<<<grid_for(n, T, 8, s->num_sms), T, 0, st>>>(s->shared, s->adj_off, s->adj, s->inst, s->cj1,
                                                                    s->cstate, s->info, ends);
        if (s->composite) {
            rc = run_comp_records(s, warm);
            if (rc != NBGS_OK) return rc;
        } else if (s->fp32)
            k_build_sweep<float><<<gb, T, 0, st>>>(Cn, n, s->inv, s->cj1, s->cj2, S, s->cgeo,
                                                   s->clev, s->prm.dt,
                                                   s->prm.beta, s->prm.mu, scene_view(s), warm, s->prev_row_off,
                                                   s->prev_j2,
                                                   s->prev_P, s->ccap, s->cstate, s->cpack, s->cmask,
                                                   (const float4*)s->vel, (SweepRec<float>*)s->srec, (float4*)s->sp,
                                                   (SweepPre<float>*)s->spre);
        else
            k_build_sweep<double><<<gb, T, 0, st>>>(Cn, n, s->inv, s->cj1, s->cj2, S, s->cgeo,
                                                    s->clev, s->prm.dt,
                                                    s->prm.beta, s->prm.mu, scene_view(s), warm, s->prev_row_off,
                                                    s->prev_j2,
                                                    s->prev_P, s->ccap, s->cstate, s->cpack, s->cmask,
                                                    (const double4_32a*)s->vel, (SweepRec<double>*)s->srec,
                                                    (double4_32a*)s->sp, (SweepPre<double>*)s->spre);
        if (s->timing) s->phase_launches[1] += 3;
        s->n_colours = -1;  // known on the device; read lazily
    } else {
        s->n_colours = 0;
    }
    if (s->timing) cudaEventRecord(s->ev[3], st);
    s->coloured = true;
    return cuda_check(s, cudaGetLastError(), "colour");
}

}  // namespace nbgs
