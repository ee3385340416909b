// Many Monte Carlo sweeps per launch with the lattice resident in shared memory (Methods,
// "Checkerboard update"; the same rule, order and random bits as the half-sweep kernels, so the
// trajectory is the same).
//
// One thread-block cluster owns one lattice: CTA c of the CS CTAs holds both sublattices of the
// planes c P .. (c + 1) P - 1 (P = L / CS) and a copy of the neighbouring CTAs' boundary planes.  A
// half-sweep reads only the CTA's own shared memory; the new words of a boundary plane are also
// stored into the neighbour's copy (distributed shared memory), and a cluster barrier separates
// half-sweeps.  A copy of sublattice q is written during q's half-sweep and read during the other's,
// so one barrier per half-sweep orders both.  The Philox draws of the next half-sweep do not depend
// on the spins: they are made between a half-sweep's arrival at the barrier and its wait.
//
// One launch per half-sweep costs 4 us for lattices this small (launch, ramp, refill of every SM from
// L2).  Here a half-sweep of a 64^3 lattice over eight CTAs takes 0.5 us: latency, of the barrier and
// of one update.  With full SMs the integer pipes bound it: 62 ALU and 26 multiply instructions per
// group of 128 spins, 45 SM cycles per 32 groups.
#include <algorithm>
#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "kernels.h"

namespace ising {

namespace {

enum ResKind : int { RES_W1, RES_W2 };  // L = 64 (rows of one word); L = 128 (two words)

struct ResArgs {
    uint4 *lat;     // replica 0
    int64_t nw4;    // uint4 per sublattice
    uint64_t seed;
    const uint64_t *seeds;  // Philox keys of the launch's lattices, or null: seed + replica
    int L, P, CS;
    uint32_t t0;
    int n;          // sweeps
    int mixed;
};

__device__ __forceinline__ uint32_t res_rank()
{
    uint32_t r;
    asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
    return r;
}

__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }

__device__ __forceinline__ uint32_t map_rank(uint32_t addr, uint32_t rank)
{
    uint32_t a;
    asm("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(addr), "r"(rank));
    return a;
}

__device__ __forceinline__ void st_cluster(uint32_t addr, const uint4 &v)
{
    asm volatile("st.shared::cluster.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
                 : "memory");
}

// x-neighbour word that is not the same word: shifted towards x - 1 (P = 0) or x + 1.  P is a
// compile-time constant of each unrolled plane: chosen at run time it took two more ALU
// operations per word.
template <int P>
__device__ __forceinline__ uint32_t res_xs(uint32_t c, uint32_t prev, uint32_t next)
{
    return P ? __funnelshift_r(c, next, 1) : __funnelshift_l(prev, c, 1);
}

// f(std::integral_constant<int, i>) for i = 0 .. N - 1
template <int N, int I = 0, class F>
__device__ __forceinline__ void res_each(F &&f)
{
    if constexpr (I < N) {
        f(std::integral_constant<int, I>{});
        res_each<N, I + 1>(f);
    }
}

// New word from the six neighbour words, the old word and its random bits.
template <int RULE>
__device__ __forceinline__ uint32_t res_word(uint32_t s, uint32_t a, uint32_t b, uint32_t c, uint32_t d, uint32_t e,
                                             uint32_t f, uint32_t rnd)
{
    const uint32_t s1 = a ^ b ^ c, c1 = maj3(a, b, c), s2 = d ^ e ^ f, c2 = maj3(d, e, f);
    const uint32_t tau = RULE == TIE_GLAUBER ? s ^ rnd : (RULE == TIE_ALWAYS ? ~s : s);
    return maj3(c1, c2, maj3(s1, s2, tau));
}

// Tie bits of the G groups grp, grp + stride, ... for sweep t and phase q: philox4x32_10 of (group, t,
// q, 0), the parts that do not depend on the group worked out first (philox_lead).  The round keys
// lie in shared memory (keys[i] = words 0 and 1 of round i) and a round is done for all groups
// together: held in registers the keys cost 18 of the 64 that 1024 threads leave, and spills.
template <int G>
__device__ __forceinline__ void res_draws(U4 (&o)[G], uint32_t grp, uint32_t stride, uint32_t t, uint32_t q,
                                          const uint2 *keys)
{
    const uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u;
    const uint2 k0 = keys[0], k1 = keys[1], k2 = keys[2];
    const uint32_t p1h = q ? __umulhi(M1, 1u) : 0u, p1l = q ? M1 : 0u;  // M1 q
    const uint32_t w0 = p1h ^ t ^ k0.x;
    const uint32_t x0 = p1l ^ k1.x, x2 = __umulhi(M0, w0) ^ k1.y, x3 = (M0 * w0) ^ k2.y;
#pragma unroll
    for (int i = 0; i < G; ++i) {
        uint32_t h0, l0, h1, l1, h2, l2, h3, l3;
        mul_hi_lo(M0, grp + (uint32_t)i * stride, h0, l0);
        mul_hi_lo(M1, h0 ^ k0.y, h1, l1);
        mul_hi_lo(M0, h1 ^ x0, h2, l2);
        mul_hi_lo(M1, l0 ^ x2, h3, l3);
        o[i].x = h3 ^ l1 ^ k2.x;
        o[i].y = l3;
        o[i].z = h2 ^ x3;
        o[i].w = l2;
    }
#pragma unroll
    for (int r = 3; r < 10; ++r) {
        const uint2 k = keys[r];
#pragma unroll
        for (int i = 0; i < G; ++i) {
            uint32_t h0, l0, h1, l1;
            mul_hi_lo(M0, o[i].x, h0, l0);
            mul_hi_lo(M1, o[i].z, h1, l1);
            o[i].x = h1 ^ o[i].y ^ k.x;
            o[i].z = h0 ^ o[i].w ^ k.y;
            o[i].y = l1;
            o[i].w = l0;
        }
    }
}

// Round keys of Philox key S into shared memory (threads 0 .. 9).
__device__ __forceinline__ void res_keys(uint2 *keys, uint64_t S)
{
    const uint32_t i = threadIdx.x;
    if (i < 10) keys[i] = make_uint2((uint32_t)S + i * 0x9E3779B9u, (uint32_t)(S >> 32) + i * 0xBB67AE85u);
}

}  // namespace

// Thread tid updates slot tid % U of the G planes zl .. zl + G - 1, zl = G (tid / U) (G and P even, so
// plane zl + i has parity i).  The other sublattice's column passes through registers.
template <int RULE, int KIND, int G, int MAXT>
__global__ void __launch_bounds__(MAXT) k_resident(const ResArgs ra)
{
    extern __shared__ __align__(16) uint4 rsm[];  // [2][P + 2][U]: planes -1 .. P of both sublattices
    __shared__ uint2 keys[10];
    constexpr int U = KIND == RES_W1 ? 16 : 64;
    const int tid = threadIdx.x, P = ra.P, L = ra.L, CS = ra.CS;
    const int c = (int)res_rank(), r = (int)blockIdx.x / CS;
    const uint64_t S = ra.seed + (uint64_t)r;
    uint4 *lat = ra.lat + 2 * (int64_t)r * ra.nw4;
    const int sub = (P + 2) * U;  // uint4 of a sublattice
    for (int q = 0; q < 2; ++q)
        for (int e = tid; e < sub; e += blockDim.x) {
            const int pl = e / U, nu = e - pl * U;
            int z = c * P + pl - 1;
            z = z < 0 ? z + L : (z >= L ? z - L : z);
            rsm[q * sub + pl * U + nu] = __ldcg(lat + (int64_t)q * ra.nw4 + (int64_t)z * U + nu);
        }
    res_keys(keys, ra.seeds ? ra.seeds[r] : S);
    const int s = tid % U, zl = G * (tid / U);
    const uint32_t grp0 = (uint32_t)((c * P + zl) * U + s);
    // first uint4 of the thread's column in a sublattice (plane zl - 1 is storage plane zl)
    const int col = zl * U + s;
    const uint32_t base = (uint32_t)__cvta_generic_to_shared(rsm);
    const uint32_t up = map_rank(base, (uint32_t)(c + 1 == CS ? 0 : c + 1));    // its plane -1 is our P - 1
    const uint32_t down = map_rank(base, (uint32_t)(c == 0 ? CS - 1 : c - 1));  // its plane P is our 0
    const bool lo = zl == 0, hi = zl + G == P;
    U4 rnd[G];
    auto draw = [&](uint32_t t, uint32_t q) {
        if (RULE != TIE_GLAUBER) return;
        res_draws<G>(rnd, grp0, U, t, q, keys);
    };
    auto half_q = [&](auto QC) {  // sublattice q; its shift direction on plane zl is q (zl is even)
        constexpr int q = decltype(QC)::value;
        const uint4 *O = rsm + (1 - q) * sub;
        uint4 *Q = rsm + q * sub;
        uint4 cm = O[col], cc = O[col + U];
        res_each<G>([&](auto I) {
            constexpr int i = decltype(I)::value, p = (q + i) & 1, np = 1 - p;
            const uint4 *pl = O + (zl + i + 1) * U;  // the plane's words
            const uint4 cp = O[col + (i + 2) * U];
            const uint4 sv = Q[col + (i + 1) * U];
            const uint4 o = make_uint4(rnd[i].x, rnd[i].y, rnd[i].z, rnd[i].w);
            uint4 nv;
            if (KIND == RES_W2) {
                // words: x, y = row 2 s; z, w = row 2 s + 1
                const uint2 *pw = reinterpret_cast<const uint2 *>(pl);
                const uint2 a = pw[(2 * s + 127) & 127], b = pw[(2 * s + 2) & 127];
                nv.x = res_word<RULE>(sv.x, cc.x, res_xs<p>(cc.x, cc.y, cc.y), a.x, cc.z, cm.x, cp.x, o.x);
                nv.y = res_word<RULE>(sv.y, cc.y, res_xs<p>(cc.y, cc.x, cc.x), a.y, cc.w, cm.y, cp.y, o.y);
                nv.z = res_word<RULE>(sv.z, cc.z, res_xs<np>(cc.z, cc.w, cc.w), cc.x, b.x, cm.z, cp.z, o.z);
                nv.w = res_word<RULE>(sv.w, cc.w, res_xs<np>(cc.w, cc.z, cc.z), cc.y, b.y, cm.w, cp.w, o.w);
            } else {
                // words: rows 4 s .. 4 s + 3 (a row is a ring of its own)
                const uint32_t *pw = reinterpret_cast<const uint32_t *>(pl);
                const uint32_t a = pw[(4 * s + 63) & 63], b = pw[(4 * s + 4) & 63];
                nv.x = res_word<RULE>(sv.x, cc.x, res_xs<p>(cc.x, cc.x, cc.x), a, cc.y, cm.x, cp.x, o.x);
                nv.y = res_word<RULE>(sv.y, cc.y, res_xs<np>(cc.y, cc.y, cc.y), cc.x, cc.z, cm.y, cp.y, o.y);
                nv.z = res_word<RULE>(sv.z, cc.z, res_xs<p>(cc.z, cc.z, cc.z), cc.y, cc.w, cm.z, cp.z, o.z);
                nv.w = res_word<RULE>(sv.w, cc.w, res_xs<np>(cc.w, cc.w, cc.w), cc.z, b, cm.w, cp.w, o.w);
            }
            Q[col + (i + 1) * U] = nv;
            if (i == 0 && lo) st_cluster(down + 16u * (uint32_t)(q * sub + (P + 1) * U + s), nv);
            if (i == G - 1 && hi) st_cluster(up + 16u * (uint32_t)(q * sub + s), nv);
            cm = cc;
            cc = cp;
        });
    };
    auto half = [&](int q) {
        if (q) half_q(std::integral_constant<int, 1>{});
        else half_q(std::integral_constant<int, 0>{});
    };
    auto first_of = [&](uint32_t t) -> uint32_t {  // sublattice updated first (Supp. Methods I B)
        if (!ra.mixed) return 0u;
        return philox4x32_10(0u, t, 5u, 0u, (uint32_t)S, (uint32_t)(S >> 32)).x & 1u;
    };
    __syncthreads();
    cluster_arrive();  // every CTA has loaded its copies before a neighbour writes into them
    uint32_t f = first_of(ra.t0);
    draw(ra.t0, f);
    cluster_wait();
#pragma unroll 1
    for (int k = 0; k < 2 * ra.n; ++k) {
        half((int)((k & 1) ? 1u - f : f));
        cluster_arrive();
        const uint32_t t = ra.t0 + (uint32_t)((k + 1) >> 1);
        if (k & 1) f = first_of(t);
        draw(t, (k & 1) ? f : 1u - f);
        cluster_wait();
    }
    for (int q = 0; q < 2; ++q)
        for (int e = tid; e < P * U; e += blockDim.x) {
            const int pl = e / U, v = e - pl * U;
            lat[(int64_t)q * ra.nw4 + (int64_t)(c * P + pl) * U + v] = rsm[q * sub + (pl + 1) * U + v];
        }
}

// ---------------------------------------------------------------------------------
// The same for lattices that need SMs of several clusters' reach: a cooperative launch in which NC
// CTAs own one lattice, P = L / NC planes each, and boundary planes travel through global memory (L2).
//
// A message is one boundary plane of one sublattice: per word the word and the step it belongs to,
// eight bytes written and read as one, so a reader polls the words themselves and no fence or flag
// follows the data.  The messages of a CTA lie in its own slab of the packed store, which holds nothing
// that is needed between the load at the start and the write-back at the end (4 U of the slab's P U
// uint4 per sublattice: P >= 4).  A thread reads the neighbour's message of the column that it
// updates itself: when it overwrites its own message of sublattice q it has received the message
// that the neighbour computed after reading the previous one, so one buffer per sublattice and
// direction suffices, also when the mixed cycle updates a sublattice twice running (the tag names
// the step of the sublattice's last update).  The next step's Philox draws, half of the work, come
// between sending and polling and cover the message's way through L2.
//
// All CTAs of a launch are co-resident (cooperative launch), every poll is bounded in wall time, and
// one that gives up sets *err = 5 and makes every CTA leave.
struct ResGArgs {
    uint4 *lat;      // first replica of the launch
    int64_t nw4;
    uint64_t seed;
    const uint64_t *seeds;  // as in ResArgs
    int P, NC;
    uint32_t t0;
    int n, mixed;
    unsigned *bar;   // two zero counters: arrivals, departures (left zero)
    int *err;
    uint64_t timeout_ns;
    int inject;      // tests: block 0 leaves out one message (1) or the first barrier (2) and the waits run out
};

__device__ __forceinline__ uint64_t res_timer_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ void msg_st(uint4 *p, uint32_t a, uint32_t b, uint32_t tag)
{
    const uint64_t x = (uint64_t)a | ((uint64_t)tag << 32), y = (uint64_t)b | ((uint64_t)tag << 32);
    asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(x), "l"(y) : "memory");
}

__device__ __forceinline__ bool msg_ld(const uint4 *p, uint32_t &a, uint32_t &b, uint32_t tag)
{
    uint64_t x, y;
    asm volatile("ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%2];" : "=l"(x), "=l"(y) : "l"(p) : "memory");
    a = (uint32_t)x;
    b = (uint32_t)y;
    return (uint32_t)(x >> 32) == tag && (uint32_t)(y >> 32) == tag;
}

// Four words of a message (two halves U apart); false when the wait gave up.
__device__ __forceinline__ bool msg_wait(const uint4 *p, int U, uint4 &v, uint32_t tag, uint64_t timeout_ns)
{
    if (msg_ld(p, v.x, v.y, tag) & msg_ld(p + U, v.z, v.w, tag)) return true;
    const uint64_t t0 = res_timer_ns();
    for (int it = 0; it < (1 << 28); ++it) {
        if (msg_ld(p, v.x, v.y, tag) & msg_ld(p + U, v.z, v.w, tag)) return true;
        if ((it & 63) == 63 && res_timer_ns() - t0 > timeout_ns) return false;
    }
    return false;
}

// Barrier number `round` (1, 2) of the launch over all its CTAs (all threads call it).  The arrivals
// add up over the two rounds; the last CTA to leave the second zeroes both counters, so the next
// launch, a replayed graph's too, finds them zero.
__device__ __forceinline__ bool grid_barrier(unsigned *bar, unsigned round, int *err, uint64_t timeout_ns)
{
    __shared__ int ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        ok = 1;
        __threadfence();
        atomicAdd(bar, 1u);
        const uint64_t t0 = res_timer_ns();
        for (int it = 0;; ++it) {
            unsigned v;
            asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(bar) : "memory");
            if (v >= round * gridDim.x) break;
            if (it >= (1 << 28) || res_timer_ns() - t0 > timeout_ns) {
                atomicExch(err, 5);
                ok = 0;
                break;
            }
        }
        if (ok && round == 2u && atomicAdd(bar + 1, 1u) == gridDim.x - 1) {
            atomicExch(bar, 0u);
            atomicExch(bar + 1, 0u);
        }
        __threadfence();
    }
    __syncthreads();
    return ok != 0;
}

// Storage of a plane in shared memory.  W4 > 0 (rows of W4 uint4): the even rows, then the odd ones,
// as in k_resident.  W4 = 0 (any other row width): the plane's words in order between a copy of the
// last row before the first and a copy of the first row after the last, so that rows y - 1 and
// y + 1 of a group, which may straddle rows, are plain offsets.
template <int W>
struct ResPlane {  // L = 64 W
    static constexpr int L = 64 * W, U = 16 * W * W;              // groups of a plane
    static constexpr int W4 = W == 4 ? 1 : (W == 8 ? 2 : 0);
    static constexpr int F = W4 > 0 ? 0 : (W + 3) / 4;            // uint4 before row 0
    static constexpr int PU = U + 2 * F;                          // uint4 of a plane
};
static int resg_plane(int W) { return 16 * W * W + (W == 4 || W == 8 ? 0 : 2 * ((W + 3) / 4)); }

// Thread tid updates group slot tid % U of the four planes zl .. zl + 3, zl = 4 (tid / U).
// Sizes are compile-time constants: with the row width at run time a group took 76 ALU and 49 multiply
// instructions at L = 512, then 74 and 40 (8.4 us per sweep, then 7.8).
template <int RULE, int W>
__global__ void __launch_bounds__(1024) k_resident_grid(const ResGArgs ra)
{
    extern __shared__ __align__(16) uint4 gsm_res[];  // [2][P][plane]
    __shared__ int s_fail;  // first step at which a poll gave up
    __shared__ uint2 keys[10];
    using RP = ResPlane<W>;
    constexpr int L = RP::L, U = RP::U, PU = RP::PU, F = RP::F, W4 = RP::W4;
    constexpr int hs = U / 2;  // W4: slots of one row parity
    constexpr bool ONE = W >= 6;  // four planes per CTA at these sizes: every thread has both boundaries
    const int tid = threadIdx.x, P = ONE ? 4 : ra.P, NC = ONE ? L / 4 : ra.NC;
    const int c = (int)blockIdx.x % NC, r = (int)blockIdx.x / NC;
    const uint64_t S = ra.seed + (uint64_t)r;
    uint4 *lat = ra.lat + 2 * (int64_t)r * ra.nw4;
    const int sub = P * PU;
    auto unit_of = [&](int sl) {  // group of a slot
        if (W4 == 0) return sl;
        const int par = sl >= hs, f = sl - par * hs, m = f / (W4 > 0 ? W4 : 1);
        return (2 * m + par) * W4 + f - m * W4;
    };
    if (tid == 0) s_fail = *(volatile int *)ra.err ? 0 : 0x7fffffff;  // an earlier launch gave up: leave at once
    for (int q = 0; q < 2; ++q)
        for (int e = tid; e < P * U; e += blockDim.x) {
            const int pl = e / U, sl = e - pl * U;
            const uint4 v = __ldcg(lat + (int64_t)q * ra.nw4 + (int64_t)(c * P + pl) * U + unit_of(sl));
            uint4 *plane = gsm_res + q * sub + pl * PU;
            plane[F + sl] = v;
            if (W4 == 0) {
                uint32_t *w = reinterpret_cast<uint32_t *>(plane) + 4 * F;
                const uint32_t vv[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                    const int k = 4 * sl + i;
                    if (k < W) w[L * W + k] = vv[i];
                    if (k >= L * W - W) w[k - L * W] = vv[i];
                }
            }
        }
    res_keys(keys, ra.seeds ? ra.seeds[r] : S);
    const int s = ONE ? tid : tid % U, zl = ONE ? 0 : 4 * (tid / U);
    const uint32_t grp0 = (uint32_t)((c * P + zl) * U + unit_of(s));
    const bool lo = ONE || zl == 0, hi = ONE || zl + 4 == P;
    const int cu = c + 1 == NC ? 0 : c + 1, cd = c == 0 ? NC - 1 : c - 1;
    // messages of CTA k, sublattice q: towards the lower neighbour at +0, the upper one at + 2 U
    auto msg = [&](int k, int q, int dir) { return lat + (int64_t)q * ra.nw4 + (int64_t)k * P * U + 2 * dir * U + s; };
    // W4: rows y - 1 and y + 1 lie in the other half of the plane
    const int yp = W4 > 0 ? (s >= hs) : 0;
    int om = 0, op = 0;
    if (W4 > 0) {
        const int f = s - yp * hs;
        om = yp ? f : hs + (f < W4 ? f + hs - W4 : f - W4);
        op = yp ? (f + W4 >= hs ? f + W4 - hs : f + W4) : hs + f;
    }
    // W4 = 0: per word of the group, the parity of its row and whether it begins or ends the row
    uint32_t rpar = 0, rfirst = 0, rlast = 0;
    if (W4 == 0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int row = (4 * s + i) / W, kw = 4 * s + i - row * W;
            rpar |= (uint32_t)(row & 1) << i;
            rfirst |= (uint32_t)(kw == 0) << i;
            rlast |= (uint32_t)(kw == W - 1) << i;
        }
    }
    __syncthreads();
    if (*(volatile int *)&s_fail == 0 || (ra.inject == 2 && blockIdx.x == 0)) return;
    // the starting state's boundary planes are the messages of step 1
    for (int q = 0; q < 2; ++q) {
        const uint4 *col = gsm_res + q * sub + F + s;
        if (lo) {
            const uint4 v = col[0];
            msg_st(msg(c, q, 0), v.x, v.y, 1u);
            msg_st(msg(c, q, 0) + U, v.z, v.w, 1u);
        }
        if (hi && !(ra.inject == 1 && blockIdx.x == 0)) {
            const uint4 v = col[(P - 1) * PU];
            msg_st(msg(c, q, 1), v.x, v.y, 1u);
            msg_st(msg(c, q, 1) + U, v.z, v.w, 1u);
        }
    }
    bool good = grid_barrier(ra.bar, 1u, ra.err, ra.timeout_ns);

    U4 rnd[4];
    auto draw = [&](uint32_t t, uint32_t q) {
        if (RULE != TIE_GLAUBER) return;
        res_draws<4>(rnd, grp0, (uint32_t)U, t, q, keys);
    };
    // one half-sweep of sublattice q as step `step`; tagO: step of the other sublattice's last update
    auto half_q = [&](auto QC, uint32_t step, uint32_t tagO, auto PB) {
        const int q = QC;  // an integral constant, or the run-time value
        const uint4 *O = gsm_res + (1 - q) * sub + zl * PU + F;
        uint4 *Q = gsm_res + q * sub + zl * PU + F;
        bool ok = true;
        uint4 cm;
        if (lo) ok = msg_wait(msg(cd, 1 - q, 1), U, cm, tagO, ra.timeout_ns);
        else cm = O[s - PU];
        uint4 cc = O[s];
        res_each<4>([&](auto I) {
            constexpr int i = decltype(I)::value, p = (decltype(PB)::value + i) & 1;
            const uint4 *pl = O + i * PU;
            uint4 cp;
            if (i == 3 && hi) ok &= msg_wait(msg(cu, 1 - q, 0), U, cp, tagO, ra.timeout_ns);
            else cp = pl[s + PU];
            const uint4 sv = Q[s + i * PU];
            const uint4 o = make_uint4(rnd[i].x, rnd[i].y, rnd[i].z, rnd[i].w);
            uint4 nv;
            if (W4 > 0) {
                const uint4 a = pl[om], b = pl[op];
                uint32_t e = p ? cc.x : cc.w;  // the row's other uint4 (W4 = 2), or this one (W4 = 1)
                if (W4 == 2) e = __shfl_xor_sync(0xffffffffu, e, 1);
                nv.x = res_word<RULE>(sv.x, cc.x, res_xs<p>(cc.x, e, cc.y), a.x, b.x, cm.x, cp.x, o.x);
                nv.y = res_word<RULE>(sv.y, cc.y, res_xs<p>(cc.y, cc.x, cc.z), a.y, b.y, cm.y, cp.y, o.y);
                nv.z = res_word<RULE>(sv.z, cc.z, res_xs<p>(cc.z, cc.y, cc.w), a.z, b.z, cm.z, cp.z, o.z);
                nv.w = res_word<RULE>(sv.w, cc.w, res_xs<p>(cc.w, cc.z, e), a.w, b.w, cm.w, cp.w, o.w);
            } else {
                const uint32_t *w = reinterpret_cast<const uint32_t *>(pl) + 4 * s;
                const uint32_t cv[4] = {cc.x, cc.y, cc.z, cc.w}, mv[4] = {cm.x, cm.y, cm.z, cm.w},
                               pv[4] = {cp.x, cp.y, cp.z, cp.w}, so[4] = {sv.x, sv.y, sv.z, sv.w},
                               ro[4] = {o.x, o.y, o.z, o.w};
                uint32_t nw[4];
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const bool pk = (((rpar >> k) + (uint32_t)(i + q)) & 1u) != 0;
                    const int d = pk ? (((rlast >> k) & 1u) ? 1 - W : 1) : (((rfirst >> k) & 1u) ? W - 1 : -1);
                    const uint32_t e = w[k + d];
                    const uint32_t x = __funnelshift_l(pk ? cv[k] : e, pk ? e : cv[k], pk ? 31 : 1);
                    nw[k] = res_word<RULE>(so[k], cv[k], x, w[k - W], w[k + W], mv[k], pv[k], ro[k]);
                }
                nv = make_uint4(nw[0], nw[1], nw[2], nw[3]);
            }
            Q[s + i * PU] = nv;
            if (W4 == 0) {
                if (4 * s < W || 4 * s + 3 >= L * W - W) {  // the copies of the first and the last row
                    uint32_t *w = reinterpret_cast<uint32_t *>(Q + i * PU);
                    const uint32_t vv[4] = {nv.x, nv.y, nv.z, nv.w};
#pragma unroll
                    for (int k = 0; k < 4; ++k) {
                        const int at = 4 * s + k;
                        if (at < W) w[L * W + at] = vv[k];
                        if (at >= L * W - W) w[at - L * W] = vv[k];
                    }
                }
            }
            if (i == 0 && lo) {
                msg_st(msg(c, q, 0), nv.x, nv.y, step);
                msg_st(msg(c, q, 0) + U, nv.z, nv.w, step);
            }
            if (i == 3 && hi) {
                msg_st(msg(c, q, 1), nv.x, nv.y, step);
                msg_st(msg(c, q, 1) + U, nv.z, nv.w, step);
            }
            cm = cc;
            cc = cp;
        });
        if (!ok) atomicMin(&s_fail, (int)step);
    };
    auto half = [&](int q, uint32_t step, uint32_t tagO) {
        using I0 = std::integral_constant<int, 0>;
        using I1 = std::integral_constant<int, 1>;
        // the sublattice as a constant too (512^3 7.79 -> 7.51 us per sweep, 448^3 8.84 -> 8.03), but not for
        // L = 256 (6.65 -> 6.81)
        if constexpr (W == 4) {
            if ((yp + q) & 1) half_q(q, step, tagO, I1{});
            else half_q(q, step, tagO, I0{});
        } else if (q) {
            if (W4 > 0 && yp == 0) half_q(I1{}, step, tagO, I1{});
            else half_q(I1{}, step, tagO, I0{});
        } else {
            if (W4 > 0 && yp != 0) half_q(I0{}, step, tagO, I1{});
            else half_q(I0{}, step, tagO, I0{});
        }
    };
    auto first_of = [&](uint32_t t) -> uint32_t {
        if (!ra.mixed) return 0u;
        return philox4x32_10(0u, t, 5u, 0u, (uint32_t)S, (uint32_t)(S >> 32)).x & 1u;
    };
    uint32_t f = first_of(ra.t0), step = 1u, last0 = 1u, last1 = 1u;
    if (good) draw(ra.t0, f);
#pragma unroll 1
    for (int k = 0; good && k < 2 * ra.n; ++k) {
        const uint32_t q = (k & 1) ? 1u - f : f;
        ++step;
        half((int)q, step, q ? last0 : last1);
        if (q) last1 = step;
        else last0 = step;
        const uint32_t t = ra.t0 + (uint32_t)((k + 1) >> 1);
        if (k & 1) f = first_of(t);
        draw(t, (k & 1) ? f : 1u - f);
        __syncthreads();
        // first step whose poll gave up: every thread reads it after the step's barrier and leaves when
        // it is at or before its own step (a thread ahead can only have written a later one)
        good = *(volatile int *)&s_fail > (int)step;
    }
    if (!good) {
        if (tid == 0) atomicExch(ra.err, 5);
        return;
    }
    if (!grid_barrier(ra.bar, 2u, ra.err, ra.timeout_ns)) return;  // every message has been read
    for (int q = 0; q < 2; ++q)
        for (int e = tid; e < P * U; e += blockDim.x) {
            const int pl = e / U, sl = e - pl * U;
            lat[(int64_t)q * ra.nw4 + (int64_t)(c * P + pl) * U + unit_of(sl)] = gsm_res[q * sub + pl * PU + F + sl];
        }
}

template <int RULE, int KIND, int G, int MAXT>
static cudaError_t launch_res(const ResArgs &ra, int R, cudaStream_t s)
{
    constexpr int U = KIND == RES_W1 ? 16 : 64;
    const int threads = ra.P * U / G;
    const size_t smem = (size_t)2 * (ra.P + 2) * U * sizeof(uint4);
    auto kern = k_resident<RULE, KIND, G, MAXT>;
    // the limit is the same whatever the plan (two CTAs per lattice need the most): another thread may launch
    // the kernel with another plan between this call and the launch
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         2 * ((KIND == RES_W1 ? 32 : 64) + 2) * U * (int)sizeof(uint4));
    if (e == cudaSuccess && ra.CS > 8) e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)(R * ra.CS));
    lc.blockDim = dim3((unsigned)threads);
    lc.dynamicSmemBytes = smem;
    lc.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)ra.CS;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    lc.attrs = at;
    lc.numAttrs = 1;
    return cudaLaunchKernelEx(&lc, kern, ra);
}

template <int RULE>
static cudaError_t res_rule(ResArgs ra, int R, int G, cudaStream_t s)
{
    switch (ra.L) {
    case 64: return G == 2 ? launch_res<RULE, RES_W1, 2, 512>(ra, R, s) : launch_res<RULE, RES_W1, 4, 256>(ra, R, s);
    case 128:
        return G == 2 ? launch_res<RULE, RES_W2, 2, 1024>(ra, R, s) : launch_res<RULE, RES_W2, 4, 1024>(ra, R, s);
    default: return cudaErrorInvalidValue;
    }
}

constexpr int RESG_MAX_SMEM = 220 * 1024;  // of every plan; the kernel's limit, as above

template <int RULE, int W>
static cudaError_t launch_resg(const ResGArgs &ra, int R, cudaStream_t s)
{
    constexpr int U = ResPlane<W>::U;
    const size_t smem = (size_t)2 * ra.P * ResPlane<W>::PU * sizeof(uint4);
    auto kern = k_resident_grid<RULE, W>;
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, RESG_MAX_SMEM);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)(R * ra.NC));
    lc.blockDim = dim3((unsigned)(ra.P * U / 4));
    lc.dynamicSmemBytes = smem;
    lc.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;
    at[0].val.cooperative = 1;
    lc.attrs = at;
    lc.numAttrs = 1;
    return cudaLaunchKernelEx(&lc, kern, ra);
}

template <int RULE>
static cudaError_t resg_rule(const ResGArgs &ra, int W, int R, cudaStream_t s)
{
    switch (W) {
    case 3: return launch_resg<RULE, 3>(ra, R, s);
    case 4: return launch_resg<RULE, 4>(ra, R, s);
    case 5: return launch_resg<RULE, 5>(ra, R, s);
    case 6: return launch_resg<RULE, 6>(ra, R, s);
    case 7: return launch_resg<RULE, 7>(ra, R, s);
    case 8: return launch_resg<RULE, 8>(ra, R, s);
    default: return cudaErrorInvalidValue;
    }
}

static cudaError_t resident_grid(const uint64_t *seeds, uint32_t *lat, int L, int R, uint64_t seed, int rule, int64_t t0, int64_t n,
                                        int cycle, int NC, unsigned *bar, int *err, double timeout_s, cudaStream_t s, int inject)
{
    const Geom g = make_geom(L);
    ResGArgs ra{};
    ra.inject = inject;
    ra.seeds = seeds;
    ra.lat = reinterpret_cast<uint4 *>(lat);
    ra.nw4 = g.nw / 4;
    ra.seed = seed;
    ra.NC = NC;
    ra.P = L / NC;
    ra.t0 = (uint32_t)t0;
    ra.n = (int)n;
    ra.mixed = cycle;
    ra.bar = bar;
    ra.err = err;
    ra.timeout_ns = (uint64_t)(timeout_s * 1e9);
    switch (rule) {
    case TIE_GLAUBER: return resg_rule<TIE_GLAUBER>(ra, g.W, R, s);
    case TIE_ALWAYS: return resg_rule<TIE_ALWAYS>(ra, g.W, R, s);
    default: return resg_rule<TIE_NEVER>(ra, g.W, R, s);
    }
}

static cudaError_t resident_cluster(const uint64_t *seeds, uint32_t *lat, int L, int R, uint64_t seed, int rule, int64_t t0, int64_t n,
                                       int cycle, int CS, int G, cudaStream_t s)
{
    const Geom g = make_geom(L);
    ResArgs ra{};
    ra.seeds = seeds;
    ra.lat = reinterpret_cast<uint4 *>(lat);
    ra.nw4 = g.nw / 4;
    ra.seed = seed;
    ra.L = L;
    ra.CS = CS;
    ra.P = L / CS;
    ra.t0 = (uint32_t)t0;
    ra.n = (int)n;
    ra.mixed = cycle;
    switch (rule) {
    case TIE_GLAUBER: return res_rule<TIE_GLAUBER>(ra, R, G, s);
    case TIE_ALWAYS: return res_rule<TIE_ALWAYS>(ra, R, G, s);
    default: return res_rule<TIE_NEVER>(ra, R, G, s);
    }
}


// Cooperative launches of this process on one device run side by side while their CTAs, counted at one
// per SM, fit the device, and wait for earlier ones otherwise: grids that were resident in part would
// wait for each other's SMs until their bounds.  Launches that are ordered one behind the other form a
// chain, as wide as its widest launch, and the chains in flight never add up to more CTAs than SMs.  (Two
// 192^3 on streams of their own: 4.5 us per sweep of both side by side, 9.0 one after the other.  Not
// while a stream is being captured: an event recorded outside cannot order a graph.  The launch of the
// graph is ordered instead.)
namespace {
struct CoopChain {
    cudaEvent_t ev = nullptr;  // end of its last launch
    cudaStream_t stream = nullptr;
    int ctas = 0;              // 0: free
    uint64_t seq = 0;
};
struct CoopDevice {
    std::mutex m;
    CoopChain chain[16];
    uint64_t seq = 0;
};
CoopDevice g_coop[64];
}  // namespace

CoopOrder::CoopOrder(cudaStream_t s, int ctas) : stream(s)
{
    cudaStreamCaptureStatus st = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(s, &st) != cudaSuccess || st != cudaStreamCaptureStatusNone) return;
    int d = -1;
    if (cudaGetDevice(&d) != cudaSuccess || d < 0 || d >= 64) return;
    dev = d;
    CoopDevice &g = g_coop[dev];
    g.m.lock();
    // an event may be queried while some other stream is being captured
    cudaStreamCaptureMode mode = cudaStreamCaptureModeRelaxed;
    cudaThreadExchangeStreamCaptureMode(&mode);
    const int sms = device_sms();
    width = std::max(1, std::min(ctas, sms));
    const int need = width;
    int busy = 0;
    auto join = [&](CoopChain &c) {  // this launch continues c
        cudaStreamWaitEvent(stream, c.ev, 0);
        width = std::max(width, c.ctas);
        busy -= c.ctas;
        c.ctas = 0;
    };
    auto oldest = [&]() -> CoopChain & {
        CoopChain *o = nullptr;
        for (CoopChain &c : g.chain)
            if (c.ctas && (!o || c.seq < o->seq)) o = &c;
        return *o;
    };
    for (CoopChain &c : g.chain) {
        if (c.ctas && cudaEventQuery(c.ev) == cudaSuccess) c.ctas = 0;
        busy += c.ctas;
    }
    cudaGetLastError();  // "not ready" is kept as the last error
    for (CoopChain &c : g.chain)
        if (c.ctas && c.stream == stream) join(c);
    while (busy + need > sms) join(oldest());
    for (slot = 0; slot < 16 && g.chain[slot].ctas; ++slot) {
    }
    if (slot == 16) {
        CoopChain &c = oldest();
        slot = (int)(&c - g.chain);
        join(c);
    }
    CoopChain &c = g.chain[slot];
    if (!c.ev && cudaEventCreateWithFlags(&c.ev, cudaEventDisableTiming) != cudaSuccess) c.ev = nullptr;
    cudaThreadExchangeStreamCaptureMode(&mode);
}

CoopOrder::~CoopOrder()
{
    if (dev < 0) return;
    CoopDevice &g = g_coop[dev];
    CoopChain &c = g.chain[slot];
    if (c.ev && cudaEventRecord(c.ev, stream) == cudaSuccess) {
        c.stream = stream;
        c.ctas = width;
        c.seq = ++g.seq;
    }
    g.m.unlock();
}

// Whether and how R lattices of size L are swept resident (host arithmetic; sms: the device's SMs).
//
// Clusters, L = 64 and 128: as many CTAs per lattice as keep the launch's CTAs within two per SM, and
// for many lattices two CTAs with more groups per thread (us per sweep, 64^3: 16 replicas 1.05 with 8
// CTAs each, 1.58 with one; 64 replicas 1.29 with 4; 512 replicas 4.9 with 2, 6.1 with one; against 8.2,
// 12.3 and 50 of the half-sweep kernel.  128^3: 6 replicas 1.33 with 16 CTAs, 1.92 with 8; 38 replicas
// 4.7 with 8, 5.7 with 2; 64 replicas 5.7 with 2, 6.7 with 8; against 12.3, 30 and 49).
//
// Grid, L = 192 .. 512: a launch holds as many lattices as its CTAs fit one per SM, P = 4, 8, ...
// planes each; the P with the least rounds x time per sweep, the time being linear in the groups of
// a CTA above a floor of latency (measured: rows of whole uint4 1.2 + 1.35e-3 per group, at least
// 3.4 us; other rows 3.5 + 2.05e-3, at least 4.9).  Per sweep: 8 x 256^3 6.6 us against 14.3 of the
// half-sweep kernel, one 512^3 7.5 against 14.8 (four: 30.1 against 39.9), 2 x 320^3 9.0 against 28.7.
//
// min_n: sweeps per call from which the load, the two grid barriers and the write-back (16 - 18 us
// a round) are earned back.
bool resident_plan(int L, int R, int sms, ResidentPlan *out)
{
    ResidentPlan p{};
    if (L == 64 || L == 128) {
        const int64_t two_per_sm = 2 * (int64_t)sms;
        if (L == 64) {
            p.ctas = R * 8 <= two_per_sm ? 8 : (R * 4 <= two_per_sm ? 4 : 2);
            p.groups = p.ctas > 2 ? 2 : 4;
        } else {
            p.ctas = R * 16 <= two_per_sm ? 16 : (R * 8 <= two_per_sm ? 8 : 2);
            p.groups = R * 16 <= sms ? 2 : 4;
        }
        p.per_launch = std::min(R, 4096);
        p.min_n = 1;
        p.us = L == 64 ? std::max(1.0, 0.3 + 0.009 * R) : std::max(1.35, 0.3 + 0.095 * R);
        p.start_us = 4.5;
        p.cluster = true;
        *out = p;
        return true;
    }
    if (L < 192 || L > 512 || L % 64 != 0) return false;
    const int W = L / 64, U = L * W / 4;
    const bool whole = W == 4 || W == 8;  // rows of whole uint4
    double best = 1e300;
    for (int P = 4; P <= L / 2; P += 4) {
        if (L % P != 0 || P * U / 4 > 1024 || L / P > sms || (W >= 6 && P != 4)) continue;
        if ((size_t)2 * P * resg_plane(W) * sizeof(uint4) > RESG_MAX_SMEM) continue;
        const int per = std::min(R, sms / (L / P));
        const int rounds = (R + per - 1) / per;
        const double us = whole ? std::max(3.4, 1.2 + 1.35e-3 * P * U) : std::max(4.9, 3.5 + 2.05e-3 * P * U);
        if (rounds * us < best) {
            best = rounds * us;
            p.us = best;
            p.start_us = 12.0 * rounds;
            p.ctas = L / P;
            p.per_launch = per;
        }
    }
    if (p.ctas == 0) return false;
    p.groups = 4;
    p.min_n = L == 256 ? 4 : (L == 512 ? (R == 1 ? 3 : (R == 2 ? 6 : 12)) : 2);
    p.cluster = false;
    *out = p;
    return true;
}

cudaError_t launch_sweeps_resident(uint32_t *lat, int L, int R, uint64_t seed, int rule, int64_t t0, int64_t n,
                                   int cycle, const ResidentPlan &p, int *err, double timeout_s, cudaStream_t s,
                                   int64_t *launches, const uint64_t *seeds, int inject)
{
    const int64_t words = 2 * make_geom(L).nw;
    unsigned *bar = reinterpret_cast<unsigned *>(err + 1);
    bool first = true;
    while (n > 0) {
        const int64_t chunk = std::min<int64_t>(n, 4096);  // bounds the length of a launch
        for (int r0 = 0; r0 < R; r0 += p.per_launch) {
            const int nr = std::min(p.per_launch, R - r0);
            uint32_t *l = lat + (int64_t)r0 * words;
            const uint64_t *sr = seeds ? seeds + r0 : nullptr;
            cudaError_t e;
            if (p.cluster) {
                e = resident_cluster(sr, l, L, nr, seed + (uint64_t)r0, rule, t0, chunk, cycle, p.ctas, p.groups, s);
            } else {
                const CoopOrder order(s, nr * p.ctas);
                e = resident_grid(sr, l, L, nr, seed + (uint64_t)r0, rule, t0, chunk, cycle, p.ctas, bar, err, timeout_s, s,
                                  first ? inject : 0);
            }
            // a device that cannot hold the clusters or the grid (a partition of the GPU) refuses the
            // first launch, before anything is enqueued
            if (e == cudaErrorInvalidClusterSize || e == cudaErrorCooperativeLaunchTooLarge ||
                e == cudaErrorLaunchOutOfResources) {
                if (first) {
                    cudaGetLastError();
                    return cudaErrorNotSupported;
                }
            }
            if (e != cudaSuccess) return e;
            first = false;
            if (launches) *launches += 1;
        }
        t0 += chunk;
        n -= chunk;
    }
    return cudaSuccess;
}

}  // namespace ising
