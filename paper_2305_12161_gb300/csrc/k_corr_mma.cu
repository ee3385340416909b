// Axis correlation sums D_a(r), and with them M and B, on the tensor cores.
//
// Along one axis the lattice is L^2 lines of L sites.  With s = +-1,
//   sum_i [s_i != s_(i + r e_a)] = (L * L^2 - S(r)) / 2,   S(r) = sum_j G[j][(j + r) mod L],
// where G[j][k] = sum over lines of s(j) s(k) is the Gram matrix of the L positions over
// the lines: a dense contraction of length L^2.  A spin is one e2m1 value (+1.0 = 0x2, -1.0 =
// 0xA, exact), block scales are all 1.0, products accumulate in fp32, and every partial sum is
// an even integer of magnitude <= L^2 <= 2^22, so the result is exact.
//
// The operands never exist in global memory: the warps of a CTA read packed lattice words,
// turn each 32-bit word into 32 nibbles (two logic operations per eight spins: the order of the
// lines inside the contraction is free, so out word j takes the bits j, j + 4, j + 8, ...) and
// write them into the shared-memory tiles (and, for off-diagonal units of line-order copies, the
// tensor-memory A tile) that tcgen05.mma reads.  At L = 2048 a measurement takes 8.7 ms against
// 21.1 with e4m3 operands staged through global memory (8.6 GB written and re-read per axis, and
// half the tensor rate); eight L = 256 replicas take 0.044 ms against 0.51 by bit counts, 512 of
// L = 64 0.04 against 0.28.  At L = 2048 the filling warps' instructions bound it: a stage of four
// products is 512 cycles of tensor work and takes about 760.
//
// Only the upper block triangle of G is computed (G is symmetric): an entry j < k stands for
// both ordered pairs, i.e. for the distances k - j and L - (k - j).  B is the sum of the three
// axes' D_a(1), and M is counted by the warps that read the z axis's words, so a measurement
// is one pass of this kernel (plus, for most L >= 512, copies of the lattice in the order it reads).
#include <algorithm>

#include "common.cuh"
#include "kernels.h"

namespace ising {

constexpr int GB_ROW = 128;                    // bytes of a position's row in a stage: 256 lines
constexpr int GB_LINES = 256;
constexpr int GB_ARRIVE = 120;                 // arrivals of a full stage, shared by its warps
constexpr int GB_SACC = 2048;                  // distance sums (largest L)
constexpr int GB_WAIT_LIMIT = 1 << 30;         // backstop on try_wait rounds (wall time comes first)

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor of tcgen05.mma for a K-major operand in 128-byte swizzled
// atoms (8 rows x 128 bytes; the 16-byte chunk c of row r stored at chunk c ^ r): start
// address, leading byte offset 16 (unused when K fits one atom row), stride 1024 bytes between
// atoms along M/N, descriptor version 1, swizzle mode 128B.  The K slice of 64 e2m1 values at
// byte offset 32 s of the atom row is addressed by starting 32 s bytes later.
__device__ __forceinline__ uint64_t umma_desc_sw128(uint32_t saddr)
{
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

// The same without swizzling, so that a row's eight 16-byte pieces lie at constant distances and the
// filling warps need no address arithmetic between them: 8 rows x 16 bytes contiguous, 128 bytes
// from one such block to the next along K, 1024 along M/N; a K slice of 64 e2m1 values starts every
// 256 bytes.
__device__ __forceinline__ uint64_t umma_desc_plain(uint32_t saddr)
{
    return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)(128 >> 4) << 16) | ((uint64_t)(1024 >> 4) << 32) |
           ((uint64_t)1 << 46);
}

// K slice q of the operand whose first row is at saddr.
template <bool PLAIN>
__device__ __forceinline__ uint64_t stage_desc(uint32_t saddr, int q)
{
    return PLAIN ? umma_desc_plain(saddr + 256 * q) : umma_desc_sw128(saddr + 32 * q);
}

// Instruction descriptor of kind::mxf4 (dense, K = 64): A and B e2m1 (bits 7 and 10), both
// K-major, N / 8 at bit 17, scales ue8m0 (bit 23), M / 128 at bit 27.
__device__ __forceinline__ uint32_t mxf4_idesc(int N)
{
    return (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | (1u << 23) | (1u << 27);
}

// D += A B of one K = 64 slice, every block scale read from tensor memory at `scale`.
__device__ __forceinline__ void mma_mxf4(uint32_t d, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t scale,
                                         uint32_t acc)
{
    asm volatile("{\n.reg .pred p;\nsetp.ne.u32 p, %4, 0;\n"
                 "tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], %1, %2, %3, [%5], [%5], p;\n}\n" ::"r"(d),
                 "l"(ad), "l"(bd), "r"(idesc), "r"(acc), "r"(scale));
}

// The same with the A operand in tensor memory: row i of the slice in lane i, its 64 values in eight
// columns from `a` on.
__device__ __forceinline__ void mma_mxf4_ta(uint32_t d, uint32_t a, uint64_t bd, uint32_t idesc, uint32_t scale,
                                            uint32_t acc)
{
    asm volatile("{\n.reg .pred p;\nsetp.ne.u32 p, %4, 0;\n"
                 "tcgen05.mma.cta_group::1.kind::mxf4.block_scale.scale_vec::2X [%0], [%1], %2, %3, [%5], [%5], p;\n}\n" ::"r"(
                     d),
                 "r"(a), "l"(bd), "r"(idesc), "r"(acc), "r"(scale));
}

// Tensor-memory columns of slot i's A tile (32 columns): beside the 256 accumulator columns of an
// off-diagonal unit, around the scales at 384 .. 415.  An A tile there is neither written to nor read
// from shared memory, and six stages fit the ring in place of four.
__device__ __forceinline__ uint32_t a_column(uint32_t slot) { return (slot < 4u ? 256u : 288u) + 32u * slot; }

// Four columns of this lane's row of an A tile, in the warp's quarter of the lanes.
__device__ __forceinline__ void tst128(uint32_t at, const uint4 &x)
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};" ::"r"(at), "r"(x.x), "r"(x.y),
                 "r"(x.z), "r"(x.w)
                 : "memory");
}

// One lane of the warp.  The compiler knows that a branch on it is taken by a single lane, which
// keeps the MMA operands in uniform registers: with `lane == 0` instead the issue loop took 1120
// cycles per stage at L = 1024, with it 835.
__device__ __forceinline__ bool elect_one()
{
    uint32_t p;
    asm volatile("{\n.reg .pred p;\nelect.sync _|p, 0xffffffff;\nselp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
    return p != 0;
}

__device__ __forceinline__ uint64_t globaltimer_ns()
{
    uint64_t t;
    asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
    return t;
}

__device__ __forceinline__ bool mbar_try(uint32_t addr, uint32_t parity)
{
    uint32_t done;
    asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
                 : "=r"(done)
                 : "r"(addr), "r"(parity)
                 : "memory");
    return done != 0;
}

// Wait for phase `parity` of an mbarrier for at most timeout_ns of wall time (and at most
// GB_WAIT_LIMIT rounds); false when it gave up.
__device__ __forceinline__ bool mbar_wait(uint32_t addr, uint32_t parity, uint64_t timeout_ns)
{
    if (mbar_try(addr, parity)) return true;
    const uint64_t t0 = globaltimer_ns();
    for (int it = 0; it < GB_WAIT_LIMIT; ++it) {
        if (mbar_try(addr, parity)) return true;
        if ((it & 255) == 255 && globaltimer_ns() - t0 > timeout_ns) return false;
    }
    return false;
}

// Transposes the 32 x 32 bit block whose row i is lane i's word (five stages, each swapping the
// off-diagonal half-blocks of size j between lanes r and r ^ j): lane i then holds bit i of
// every row.  What depends on the lane (byte selectors, rotations, masks) is worked out once: a
// stage is a shuffle and a byte permute, or a shuffle, a rotation and a select.
struct Transpose32 {
    uint32_t sel16, sel8, rot4, rot2, rot1, keep4, keep2, keep1;
    __device__ explicit Transpose32(int lane)
    {
        sel16 = (lane & 16) ? 0x3276u : 0x5410u;
        sel8 = (lane & 8) ? 0x3715u : 0x6240u;
        rot4 = (lane & 4) ? 28u : 4u;
        rot2 = (lane & 2) ? 30u : 2u;
        rot1 = (lane & 1) ? 31u : 1u;
        keep4 = (lane & 4) ? 0xF0F0F0F0u : 0x0F0F0F0Fu;
        keep2 = (lane & 2) ? 0xCCCCCCCCu : 0x33333333u;
        keep1 = (lane & 1) ? 0xAAAAAAAAu : 0x55555555u;
    }
    __device__ __forceinline__ static uint32_t part(uint32_t v, int j, uint32_t rot, uint32_t keep)
    {
        const uint32_t t = __shfl_xor_sync(0xffffffffu, v, j);
        return (v & keep) | (__funnelshift_l(t, t, rot) & ~keep);
    }
    __device__ __forceinline__ uint32_t operator()(uint32_t v) const
    {
        v = __byte_perm(v, __shfl_xor_sync(0xffffffffu, v, 16), sel16);
        v = __byte_perm(v, __shfl_xor_sync(0xffffffffu, v, 8), sel8);
        v = part(v, 4, rot4, keep4);
        v = part(v, 2, rot2, keep2);
        return part(v, 1, rot1, keep1);
    }
};

// The 32 spins of one word as e2m1 values (32 lines of one position): nibble m of out word j is
// bit 4 m + j, sign bit set for a down spin.
__device__ __forceinline__ uint4 expand_e2m1(uint32_t v)
{
    const uint32_t S = 0x88888888u, P = 0xAAAAAAAAu;
    return make_uint4(((v << 3) & S) ^ P, ((v << 2) & S) ^ P, ((v << 1) & S) ^ P, (v & S) ^ P);
}

__device__ __forceinline__ void sts128(uint32_t addr, const uint4 &v)
{
    asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
                 : "memory");
}

// ---------------------------------------------------------------------------------
// Line order for L >= 512 (the x axis for multiples of 128, all three for multiples of 256), where each
// word is read by several CTAs: per axis a copy of the packed
// lattice, N / 8 bytes, in which uint4 (2 c + h) L + p holds half h of the 256 lines of chunk c
// at position p, so that a warp of 32 positions reads 512 consecutive bytes.  Read from the
// packed store the words of 32 positions lie 128 bytes (y) or a plane (z) apart: at L = 2048 a
// measurement took 17.6 ms that way and 13.4 with the copies (and their 1 ms) otherwise unchanged.

// x axis: the lines are rows (row = y + L z), so their bits are transposed; half h holds the bundles
// 32 (4 h + j) .. + 31 of the chunk's rows.  A CTA takes one chunk and four word columns: warp b reads
// bundle b's rows and transposes the eight 32 x 32 bit blocks in registers.  Bound by DRAM: N / 8 bytes
// in, N / 8 out.  The word columns are the fast grid index, so that the CTAs that share a row's sectors
// run together: at L = 2048 1.32 -> 0.52 ms against the chunks as the fast index, where a sector's other
// half was read 16384 CTAs later (the whole measurement 10.79 -> 9.97 ms).
// In shared memory the even positions come first, nine words apart, the odd ones 16 banks further: writes
// (lanes two positions apart) and reads (lanes one position apart) are then both free of conflicts.
__global__ void __launch_bounds__(256) k_lines_x(const uint32_t *lat, Geom g, uint32_t *T, int64_t rep_words)
{
    __shared__ uint32_t sm[256 * 9 + 16];
    const int L = g.L, W = g.W;
    const int lane = threadIdx.x & 31, b = threadIdx.x >> 5;
    const int kw0 = 4 * blockIdx.x, c = blockIdx.y, r = blockIdx.z;
    const int nkw = min(4, W - kw0);
    const uint32_t *S0 = lat + 2 * (int64_t)r * g.nw, *S1 = S0 + g.nw;
    const uint32_t row = 256u * (uint32_t)c + 32u * (uint32_t)b + (uint32_t)lane;
    const uint32_t z = row / (uint32_t)L, y = row - z * (uint32_t)L;
    const bool odd = (y + z) & 1u;
    const int64_t at = (int64_t)row * W + kw0;
    const Transpose32 tr(lane);
    uint32_t v0[4] = {0, 0, 0, 0}, v1[4] = {0, 0, 0, 0};
    if (W % 4 == 0) {
        const uint4 a = __ldg(reinterpret_cast<const uint4 *>(S0 + at));
        const uint4 d = __ldg(reinterpret_cast<const uint4 *>(S1 + at));
        v0[0] = a.x; v0[1] = a.y; v0[2] = a.z; v0[3] = a.w;
        v1[0] = d.x; v1[1] = d.y; v1[2] = d.z; v1[3] = d.w;
    } else {
#pragma unroll
        for (int i = 0; i < 4; ++i)
            if (i < nkw) {
                v0[i] = __ldg(S0 + at + i);
                v1[i] = __ldg(S1 + at + i);
            }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        const uint32_t e = tr(odd ? v1[i] : v0[i]);  // x = 2 (32 kw + lane)
        const uint32_t o = tr(odd ? v0[i] : v1[i]);  // x + 1
        sm[(32 * i + lane) * 9 + b] = e;
        sm[(128 + 32 * i + lane) * 9 + 16 + b] = o;
    }
    __syncthreads();
    const int p = threadIdx.x;  // position 64 kw0 + p: both halves of its 256 lines
    if (p >= 64 * nkw) return;
    const uint32_t *v = sm + (p & 1) * (128 * 9 + 16) + (p >> 1) * 9;
    uint4 *dst = reinterpret_cast<uint4 *>(T + (int64_t)r * rep_words) + (int64_t)c * 2 * L + 64 * kw0 + p;
    dst[0] = make_uint4(v[0], v[1], v[2], v[3]);
    dst[L] = make_uint4(v[4], v[5], v[6], v[7]);
}

// y (blockIdx.z even) and z axes, L a multiple of 256: chunk c = a W4 + k4 is the uint4 k4 of the rows
// with other coordinate a, half pi the sites x = 2k + pi.  A CTA takes 32 positions of one a.
__global__ void __launch_bounds__(256) k_lines_yz(const uint32_t *lat, Geom g, uint32_t *T, int64_t rep_words)
{
    __shared__ uint4 sm[2][8 * 33];
    const int L = g.L, W4 = g.W / 4;
    const int p0 = 32 * blockIdx.x, a = blockIdx.y, r = blockIdx.z >> 1, axis = 1 + (blockIdx.z & 1);
    const uint4 *S0 = reinterpret_cast<const uint4 *>(lat + 2 * (int64_t)r * g.nw), *S1 = S0 + g.nw / 4;
    const int t = threadIdx.x, n = 32 * W4;
    if (t < n) {
        const int i = t / W4, k = t - i * W4, p = p0 + i;
        const int64_t at = (axis == 1 ? (int64_t)a * L + p : (int64_t)p * L + a) * W4 + k;
        const bool odd = (p + a) & 1;
        sm[odd][k * 33 + i] = __ldg(S0 + at);
        sm[!odd][k * 33 + i] = __ldg(S1 + at);
    }
    __syncthreads();
    if (t < n) {
        const int k = t >> 5, i = t & 31;
        uint4 *dst = reinterpret_cast<uint4 *>(T + (int64_t)r * rep_words + (int64_t)axis * 2 * g.nw) +
                     ((int64_t)(a * W4 + k) * 2) * L + p0 + i;
        dst[0] = sm[0][k * 33 + i];
        dst[L] = sm[1][k * 33 + i];
    }
}

// ---------------------------------------------------------------------------------
// Work items.  The L positions form super-tiles of 256 (the last may be short).  A unit is either
// the diagonal block of a super-tile (its rows filled once; MMAs of rows 0..127 against all
// columns and of rows 128..255 against columns 128..) or a tile of 128 rows against a later
// super-tile.  An item is (replica, axis, slice of the lines, unit); the CTAs are persistent and
// take items in that order, so the CTAs running together read the same lines.
struct GramArgs {
    const uint32_t *lat, *lines;  // lines: copies in line order (x only unless L % 256 == 0), or null
    int64_t rep_words;            // words of one replica's copies
    int64_t *rec;
    int64_t RL, nw;            // record length; words per sublattice
    int L, W;
    int nsb, nunits, nitems;
    int split_x, split_yz;     // slices of the lines: x axis, y and z axes
    int nrep;
    int stage_bytes, nst;      // ring of stages
    int ncols, scale_col;      // tensor memory: columns allocated, first of the 32 scale columns
    int *err;
    uint64_t timeout_ns;
    int inject;
};

struct GramUnit {
    int j0, s0;  // first row of the A tile, first position of the B super-tile
    int ra, rb;  // rows filled for A (0: A is part of B) and for B
};

__device__ __forceinline__ GramUnit gram_unit(int u, int nsb, int L)
{
    GramUnit m;
    if (u < nsb) {
        m.j0 = m.s0 = 256 * u;
        m.ra = 0;
    } else {
        u -= nsb;
        int bj = 0;
        while (u >= nsb - 1 - bj / 2) {
            u -= nsb - 1 - bj / 2;
            ++bj;
        }
        m.j0 = 128 * bj;
        m.s0 = 256 * (bj / 2 + 1 + u);
        m.ra = 128;
    }
    m.rb = min(256, L - m.s0);
    return m;
}

// Readers: the eight words (256 lines) of this lane's share of one stage, for the stages
// first, first + step, ... (chunks of 256 lines).  All addresses advance by additions.

// y or z axis, rows of whole uint4 (W a multiple of 4): word pi * 4 + i is word kw + i of the row of
// position p at the other coordinate a, of the sublattice that holds the sites x = 2k + pi there;
// a chunk is four words of each.  The two sublattices swap roles whenever a advances.
struct ReadYZ4 {
    const uint4 *e, *o;  // next words of pi = 0 and pi = 1
    int k4, W4, step;
    int64_t da;          // uint4 from the end of one a's row to the next a's
    __device__ ReadYZ4(const uint32_t *S0, const uint32_t *S1, int L, int W, int axis, int p, int c, int st)
    {
        W4 = W / 4;
        step = st;
        const int a = c / W4;
        k4 = c - a * W4;
        const int64_t at = (axis == 1 ? (int64_t)a * L + p : (int64_t)p * L + a) * W4 + k4;
        da = axis == 1 ? (int64_t)(L - 1) * W4 : 0;
        const bool odd = (p + a) & 1;
        e = reinterpret_cast<const uint4 *>(odd ? S1 : S0) + at;
        o = reinterpret_cast<const uint4 *>(odd ? S0 : S1) + at;
    }
    __device__ __forceinline__ void next(uint32_t v[8])
    {
        const uint4 s = __ldg(e), t = __ldg(o);
        v[0] = s.x; v[1] = s.y; v[2] = s.z; v[3] = s.w;
        v[4] = t.x; v[5] = t.y; v[6] = t.z; v[7] = t.w;
        e += step;
        o += step;
        k4 += step;
        while (k4 >= W4) {
            k4 -= W4;
            const uint4 *x = e + da;
            e = o + da;
            o = x;
        }
    }
};

// The same for other row widths: word column 4 c + i = a W + kw (a from a multiply by 2^32 / W,
// exact for the columns of these sizes: below 2^16, W <= 32).
struct ReadYZ1 {
    const uint32_t *S0, *S1;
    int L, W, axis, p, c, step;
    uint32_t inv;
    __device__ ReadYZ1(const uint32_t *s0, const uint32_t *s1, int l, int w, int ax, int pos, int c0, int st)
        : S0(s0), S1(s1), L(l), W(w), axis(ax), p(pos), c(c0), step(st)
    {
        inv = (uint32_t)((0x100000000ull + (uint32_t)w - 1) / (uint32_t)w);
    }
    __device__ __forceinline__ void next(uint32_t v[8])
    {
        const uint32_t ci = 4u * (uint32_t)c;
        int a = W == 1 ? (int)ci : (int)__umulhi(ci, inv);
        int kw = (int)ci - a * W;
        uint32_t s[4], t[4];
        if (axis == 2) {  // the four words are consecutive
            const int64_t at = (int64_t)p * L * W + ci;
            const uint4 x = __ldg(reinterpret_cast<const uint4 *>(S0 + at));
            const uint4 y = __ldg(reinterpret_cast<const uint4 *>(S1 + at));
            s[0] = x.x; s[1] = x.y; s[2] = x.z; s[3] = x.w;
            t[0] = y.x; t[1] = y.y; t[2] = y.z; t[3] = y.w;
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            if (axis == 1) {
                const int64_t at = ((int64_t)a * L + p) * W + kw;
                s[i] = __ldg(S0 + at);
                t[i] = __ldg(S1 + at);
            }
            const bool odd = (p + a) & 1;
            v[i] = odd ? t[i] : s[i];
            v[4 + i] = odd ? s[i] : t[i];
            if (++kw == W) {
                kw = 0;
                ++a;
            }
        }
        c += step;
    }
};

// An axis in line order.
struct ReadT {
    const uint4 *q;
    int64_t dq;
    int L;
    __device__ ReadT(const uint32_t *T, int l, int p, int c, int step) : L(l)
    {
        q = reinterpret_cast<const uint4 *>(T) + (int64_t)c * 2 * L + p;
        dq = (int64_t)step * 2 * L;
    }
    __device__ __forceinline__ void next(uint32_t v[8])
    {
        const uint4 s = __ldg(q), t = __ldg(q + L);
        v[0] = s.x; v[1] = s.y; v[2] = s.z; v[3] = s.w;
        v[4] = t.x; v[5] = t.y; v[6] = t.z; v[7] = t.w;
        q += dq;
    }
};

// x axis of the packed lattice: word kw of both sublattices of the rows 256 c + 32 (b0 + i) + lane;
// word 2 i + pi is bundle b0 + i's sites x = 2k + pi (still to be transposed).
struct ReadXL {
    const uint32_t *S0, *S1;
    int64_t at, dat;
    int L, W, dy, y[4];
    uint32_t odd, dodd;  // bit i: parity of z of bundle b0 + i's row
    __device__ ReadXL(const uint32_t *s0, const uint32_t *s1, int l, int w, int kw, int b0, int lane, int c, int step)
        : S0(s0), S1(s1), L(l), W(w)
    {
        const int row = 256 * c + 32 * b0 + lane;
        at = (int64_t)row * W + kw;
        dat = (int64_t)256 * step * W;
        odd = 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int z = (row + 32 * i) / L;
            y[i] = row + 32 * i - z * L;
            odd |= (uint32_t)(z & 1) << i;
        }
        dy = (256 * step) % L;
        dodd = ((256 * step) / L) & 1 ? 15u : 0u;
    }
    __device__ __forceinline__ void next(uint32_t v[8])
    {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const uint32_t a = __ldg(S0 + at + 32 * i * W), b = __ldg(S1 + at + 32 * i * W);
            const bool o = ((uint32_t)y[i] ^ (odd >> i)) & 1u;
            v[2 * i] = o ? b : a;
            v[2 * i + 1] = o ? a : b;
            y[i] += dy;
            if (y[i] >= L) {
                y[i] -= L;
                odd ^= 1u << i;
            }
        }
        odd ^= dodd;
        at += dat;
    }
};

// What a warp does for its stages of one item.  The next stage's words are loaded and the present
// one's are expanded in registers before the wait for the slot, so that between the slot's release
// and its refill there are only the shared-memory stores: the ring holds four 48 KB stages, 2048
// cycles of products, and the time round it bounds the kernel.  Returns false when a wait gave up.
struct Fill {
    uint32_t ring, full0, empty0;  // shared addresses
    int nst, stage_bytes, arrive;
    uint64_t timeout_ns;
    int skip;                      // stage whose arrival is left out (failure injection), -1: none
};

template <class Read, class Expand, class Put>
__device__ __forceinline__ bool fill_stages(const Fill &f, uint32_t g0, int set, int nsets, int n, Read &rd,
                                            Expand expand, Put put)
{
    const int lane = threadIdx.x & 31;
    uint32_t v[8];
    if (set < n) rd.next(v);
    int slot = (int)((g0 + (uint32_t)set) % (uint32_t)f.nst);
    uint32_t phase = ((g0 + (uint32_t)set) / (uint32_t)f.nst) & 1u;
#pragma unroll 1
    for (int s = set; s < n; s += nsets) {
        uint4 x[8];
        expand(v, x);
        if (s + nsets < n) rd.next(v);
        // the slot's previous use was consumed (a barrier that has completed no phase passes parity 1)
        const bool ok = mbar_wait(f.empty0 + 8u * (uint32_t)slot, phase ^ 1u, f.timeout_ns);
        if (!__all_sync(0xffffffffu, ok)) return false;  // the warp leaves together
        put((uint32_t)slot, x);
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        __syncwarp();
        if (lane == 0 && s != f.skip)
            asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;" ::"r"(f.full0 + 8u * (uint32_t)slot),
                         "r"(f.arrive)
                         : "memory");
        slot += nsets;
        if (slot >= f.nst) {
            slot -= f.nst;
            phase ^= 1u;
        }
    }
    return true;
}

// The same with the words of the next AHEAD stages under way and the expansion after the wait
// (put(slot, v) expands and stores): for the ring of six 32 KB stages, 3072 cycles of products, where the
// loads' latency shows before the time from a slot's release to its refill.  It is the filling warps'
// rate that binds there: at L = 2048 the products take 5.4 ms, and the kernel 8.5 with them left out
// and 6.0 with the filling left out.  Whole measurement: 9.97 ms with the loop above; 9.11 with
// two stages ahead, 8.97 without the swizzle, 8.72 with three, 8.73 with four.
template <int AHEAD, class Read, class Put>
__device__ __forceinline__ bool fill_stages_ahead(const Fill &f, uint32_t g0, int set, int nsets, int n, Read &rd,
                                                  Put put)
{
    const int lane = threadIdx.x & 31;
    uint32_t v[AHEAD][8];
#pragma unroll
    for (int a = 0; a < AHEAD; ++a)
        if (set + a * nsets < n) rd.next(v[a]);
    int slot = (int)((g0 + (uint32_t)set) % (uint32_t)f.nst);
    uint32_t phase = ((g0 + (uint32_t)set) / (uint32_t)f.nst) & 1u;
#pragma unroll 1
    for (int s = set; s < n;) {
#pragma unroll
        for (int a = 0; a < AHEAD; ++a) {
            if (s >= n) break;
            const bool ok = mbar_wait(f.empty0 + 8u * (uint32_t)slot, phase ^ 1u, f.timeout_ns);
            if (!__all_sync(0xffffffffu, ok)) return false;  // the warp leaves together
            put((uint32_t)slot, v[a]);
            if (s + AHEAD * nsets < n) rd.next(v[a]);
            asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
            __syncwarp();
            if (lane == 0 && s != f.skip)
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;" ::"r"(f.full0 + 8u * (uint32_t)slot),
                             "r"(f.arrive)
                             : "memory");
            slot += nsets;
            if (slot >= f.nst) {
                slot -= f.nst;
                phase ^= 1u;
            }
            s += nsets;
        }
    }
    return true;
}

// One CTA: the first PW warps fill the stages and afterwards read the accumulators, the last two
// warps issue the MMAs, one stage each in turn: while one's products run, it commits them and the other
// waits for its stage (four 512^3 0.28 -> 0.26 ms; at L = 2048, where the filling warps bind, nothing
// changed).  The turn passes through an mbarrier between tcgen05 fences, so
// the products reach the accumulators in the order of the stages.  A stage holds 256 lines of every row of the unit; the (ra + rb) / 32
// warps of a set fill it, one row per lane, and as many sets as the PW warps hold work on successive
// stages.  Each stage is written once and read by 4 (off-diagonal) or 8 MMAs of 128 x N x 64.
//
// Every wait is bounded (timeout_ns of %globaltimer).  A wait that gives up clears `flag`, every
// role leaves its loop, *err is set and nothing of the item is added to the records.  The MMA
// thread commits what it issued to `done` and waits for it before the tensor memory is released;
// if that arrival does not come either, *err = 2 and the tensor memory is kept rather than freed
// under a running MMA.
//
// READS: which readers the instantiation holds (fewer keep more warps within the registers).
// MINB CTAs share an SM.
enum GramReads : int { GR_SMALL, GR_T, GR_XL, GR_ANY };  // XL + YZ1; T alone; XL + YZ4; XL or T, and YZ1

template <int PW, int MINB, int READS>
__global__ void __launch_bounds__(32 * (PW + 2), MINB) k_gram_bits(const GramArgs ga)
{
    constexpr int GB_THREADS = 32 * (PW + 2);
    constexpr bool TA = READS == GR_T;  // A tiles in tensor memory
    extern __shared__ __align__(1024) uint8_t gsm[];
    __shared__ int sacc[GB_SACC];
    __shared__ __align__(8) uint64_t full[8], empty[8], turn[2], done;
    __shared__ uint32_t tmem_holder;
    __shared__ int flag, mma_pending, pops[2];  // up spins of the z axis's words, by item parity

    const int L = ga.L, W = ga.W, H = L / 2;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const uint32_t ring = (smem_u32(gsm) + 1023u) & ~1023u;
    const int nst = ga.nst;

    for (int i = tid; i < L; i += GB_THREADS) sacc[i] = 0;
    if (warp == PW) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(&tmem_holder)),
                     "r"(ga.ncols));
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (tid == 0) {
        for (int i = 0; i < nst; ++i) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&full[i])), "r"(GB_ARRIVE));
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&empty[i])));
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&turn[0])));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_u32(&turn[1])));
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 2;" ::"r"(smem_u32(&done)));
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        flag = 1;
        mma_pending = 0;
        pops[0] = pops[1] = 0;
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = tmem_holder;
    const uint32_t scale = tmem + (uint32_t)ga.scale_col;
    if (warp < 4) {  // every block scale is 1.0 (ue8m0 0x7F) whatever its place in the 32 columns
        const uint32_t one4 = 0x7F7F7F7Fu;
        const uint32_t at = scale + ((uint32_t)(32 * warp) << 16);
#pragma unroll
        for (int i = 0; i < 4; ++i)
            asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %1, %1, %1, %1, %1, %1, %1};" ::"r"(at + 8 * i),
                         "r"(one4));
        asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    pdl_enter();  // what precedes touches no global memory and overlaps the previous kernel's end

    const int nk = (int)((int64_t)L * L / GB_LINES);
    uint32_t g0 = 0;     // stages used by earlier items (ring position and phase)
    uint32_t nitem = 0;  // items done: phase of `done`
    uint32_t nturn = 0;  // turns this issuer has waited for: phase of its `turn`
    for (int item = blockIdx.x; item < ga.nitems; item += gridDim.x, ++nitem) {
        const int items_x = ga.nrep * ga.split_x * ga.nunits, items_y = ga.nrep * ga.split_yz * ga.nunits;
        const int axis = item < items_x ? 0 : (item < items_x + items_y ? 1 : 2);
        const int split = axis == 0 ? ga.split_x : ga.split_yz;
        int rest = item - (axis == 0 ? 0 : (axis == 1 ? items_x : items_x + items_y));
        const GramUnit un = gram_unit(rest % ga.nunits, ga.nsb, L);
        rest /= ga.nunits;
        const int r = rest / split, sl = rest - r * split;
        const int c0 = (int)((int64_t)nk * sl / split), c1 = (int)((int64_t)nk * (sl + 1) / split);
        const int n = c1 - c0;
        const uint32_t *S0 = ga.lat + 2 * (int64_t)r * ga.nw, *S1 = S0 + ga.nw;
        const bool bad_first = ga.inject && blockIdx.x == 0 && nitem == 0;

        if (warp < PW) {
            const int wps = (un.ra + un.rb) / 32;  // warps of a set: 2, 4, 6, 8, 10 or 12
            // at most nst sets: a set that moves on to stage s + nsets then finds the slot's phase at
            // most one behind the one it waits for, which the parity tells apart
            const int nsets = min(PW / wps, nst);
            const int set = warp / wps, ws = warp - set * wps;
            if (set < nsets) {
                const Fill fl{ring, smem_u32(full), smem_u32(empty), nst, ga.stage_bytes, GB_ARRIVE / wps,
                              ga.timeout_ns, bad_first && ws == 0 ? 0 : -1};
                int m = 0;
                const bool count_m = axis == 2 && un.ra == 0;
                bool ok;
                if (READS != GR_T && axis == 0 && (READS != GR_ANY || ga.lines == nullptr)) {
                    // this warp's share is word column kw and the bundles b0 .. b0 + 3 of the 64 rows
                    // (positions) of warps ws & ~1 and ws | 1
                    const int wr = 64 * (ws >> 1);
                    const bool xA = wr >= un.rb;
                    const int xr = xA ? wr - un.rb : wr;  // first of the 64 rows in its region
                    const int kw = ((xA ? un.j0 : un.s0) + xr) >> 6, b0 = 4 * (ws & 1);
                    const Transpose32 tr(lane);
                    ReadXL rd(S0, S1, L, W, kw, b0, lane, c0 + set, nsets);
                    ok = fill_stages(
                        fl, g0, set, nsets, n, rd,
                        [&](uint32_t v[8], uint4 x[8]) {
#pragma unroll
                            for (int i = 0; i < 8; ++i) x[i] = expand_e2m1(tr(v[i]));
                        },
                        [&](uint32_t slot, uint4 x[8]) {
                            const uint32_t base = ring + slot * (uint32_t)fl.stage_bytes;
#pragma unroll
                            for (int i = 0; i < 8; ++i) {  // bundle b0 + i / 2, positions 64 kw + 2 lane + (i & 1)
                                const uint32_t rr = (uint32_t)(xr + 2 * lane + (i & 1));
                                sts128(base + (xA ? 32768u : 0u) + rr * GB_ROW +
                                           ((((uint32_t)(b0 + (i >> 1))) ^ (rr & 7u)) << 4),
                                       x[i]);
                            }
                        });
                } else {
                    // this lane's row: B rows first, then (off-diagonal units) the A rows 32 KB further on
                    const int f = 32 * ws + lane;
                    const bool isA = f >= un.rb;
                    const int ri = isA ? f - un.rb : f;
                    const int p = isA ? un.j0 + ri : un.s0 + ri;
                    const uint32_t row_off = (isA ? 32768u : 0u) + (uint32_t)ri * GB_ROW + (uint32_t)((ri & 7) << 4);
                    auto expand = [&](uint32_t v[8], uint4 x[8]) {
#pragma unroll
                        for (int i = 0; i < 8; ++i) x[i] = expand_e2m1(v[i]);
                        if (count_m)
#pragma unroll
                            for (int i = 0; i < 8; ++i) m += __popc(v[i]);
                    };
                    auto put = [&](uint32_t slot, uint4 x[8]) {
                        const uint32_t at = ring + slot * (uint32_t)fl.stage_bytes + row_off;
#pragma unroll
                        for (int i = 0; i < 8; ++i) sts128(at ^ (uint32_t)(i << 4), x[i]);
                    };
                    if (TA) {
                        ReadT rd(ga.lines + (int64_t)r * ga.rep_words + (int64_t)axis * 2 * ga.nw, L, p, c0 + set, nsets);
                        const uint32_t off = (uint32_t)(ri >> 3) * 1024u + (uint32_t)(ri & 7) * 16u;
                        ok = fill_stages_ahead<3>(fl, g0, set, nsets, n, rd, [&](uint32_t slot, uint32_t v[8]) {
                            if (count_m)
#pragma unroll
                                for (int i = 0; i < 8; ++i) m += __popc(v[i]);
                            if (32 * ws >= un.rb) {  // rb is 256: A rows 32 (warp % 4) .. + 31
                                const uint32_t at = tmem + a_column(slot) + ((uint32_t)(32 * (warp & 3)) << 16);
                                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                                for (int i = 0; i < 8; ++i) tst128(at + 4u * i, expand_e2m1(v[i]));
                                asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
                                asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                            } else {
                                const uint32_t at = ring + slot * (uint32_t)fl.stage_bytes + off;
#pragma unroll
                                for (int i = 0; i < 8; ++i) sts128(at + (uint32_t)(i << 7), expand_e2m1(v[i]));
                            }
                        });
                    } else if (READS == GR_ANY && axis == 0) {
                        ReadT rd(ga.lines + (int64_t)r * ga.rep_words + (int64_t)axis * 2 * ga.nw, L, p, c0 + set, nsets);
                        ok = fill_stages(fl, g0, set, nsets, n, rd, expand, put);
                    } else if (READS == GR_XL) {
                        ReadYZ4 rd(S0, S1, L, W, axis, p, c0 + set, nsets);
                        ok = fill_stages(fl, g0, set, nsets, n, rd, expand, put);
                    } else {
                        ReadYZ1 rd(S0, S1, L, W, axis, p, c0 + set, nsets);
                        ok = fill_stages(fl, g0, set, nsets, n, rd, expand, put);
                    }
                }
                if (!ok) *(volatile int *)&flag = 0;
                if (count_m) {
#pragma unroll
                    for (int o = 16; o > 0; o >>= 1) m += __shfl_xor_sync(0xffffffffu, m, o);
                    if (lane == 0) atomicAdd(&pops[nitem & 1u], m);
                }
            }
        } else if (elect_one()) {  // MMA issuer w: the item's stages s with s % 2 == w
            const int w = warp - PW;
            const uint32_t id0 = mxf4_idesc(un.rb);
            const bool two = un.ra == 0 && un.rb > 128;
            const uint32_t id1 = mxf4_idesc(two ? un.rb - 128 : 64);
            int slot = (int)((g0 + (uint32_t)w) % (uint32_t)nst);
            uint32_t phase = ((g0 + (uint32_t)w) / (uint32_t)nst) & 1u;
            bool issued = false, ok = true;
            for (int s = w; s < n; s += 2) {
                ok = mbar_wait(smem_u32(&full[slot]), phase, ga.timeout_ns);
                if (ok && s > 0) {
                    ok = mbar_wait(smem_u32(&turn[w]), nturn & 1u, ga.timeout_ns);
                    ++nturn;
                }
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
                const uint32_t base = ring + (uint32_t)slot * (uint32_t)ga.stage_bytes;
                const uint32_t abase = un.ra ? base + 32768u : base;
                if (TA && un.ra) {  // the branch outside the loop: inside, a measurement at L = 2048 took 0.55 ms more
#pragma unroll
                    for (int q = 0; q < GB_ROW / 32; ++q)
                        mma_mxf4_ta(tmem, tmem + a_column((uint32_t)slot) + 8u * q, stage_desc<TA>(base, q), id0,
                                    scale, (s > 0 || q > 0) ? 1u : 0u);
                } else {
#pragma unroll
                    for (int q = 0; q < GB_ROW / 32; ++q)
                        mma_mxf4(tmem, stage_desc<TA>(abase, q), stage_desc<TA>(base, q), id0, scale,
                                 (s > 0 || q > 0) ? 1u : 0u);
                }
                if (two) {
#pragma unroll
                    for (int q = 0; q < GB_ROW / 32; ++q)
                        mma_mxf4(tmem + 256u, stage_desc<TA>(base + 16384u, q), stage_desc<TA>(base + 16384u, q), id1,
                                 scale, (s > 0 || q > 0) ? 1u : 0u);
                }
                issued = true;
                if (s + 1 < n) {
                    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
                    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&turn[w ^ 1])) : "memory");
                }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                    smem_u32(&empty[slot])));
                slot += 2;
                if (slot >= nst) {
                    slot -= nst;
                    phase ^= 1u;
                }
            }
            if (!ok) *(volatile int *)&flag = 0;
            // `done` completes with both issuers' arrivals: a commit covers every MMA issued before it
            if (issued)
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                    smem_u32(&done)));
            else
                asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(&done)) : "memory");
            // the other issuer may spend two bounded waits first, and one more bounded window passes before
            // the tensor memory is declared still in use
            if (!mbar_wait(smem_u32(&done), nitem & 1u, 3 * ga.timeout_ns)) {
                *(volatile int *)&flag = 0;
                mma_pending = 1;
            }
        }
        __syncwarp();
        __syncthreads();
        if (!*(volatile int *)&flag) break;
        if (warp < PW) {
            // warp w reads tensor-memory lanes 32 (w % 4) .. + 31 and every (PW / 4)-th group of 16 columns
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const int row0 = 32 * (warp & 3) + lane;
            const int ncol = un.rb, ncol1 = (un.ra == 0 && un.rb > 128) ? un.rb - 128 : 0;
#pragma unroll 1
            for (int cc = 16 * (warp >> 2); cc < ncol + ncol1; cc += 4 * PW) {
                const bool second = cc >= ncol;
                const int col = second ? cc - ncol + 256 : cc;
                const int j = un.j0 + row0 + (second ? 128 : 0);
                const int k0 = second ? un.s0 + 128 + cc - ncol : un.s0 + cc;
                uint32_t v[16];
                const uint32_t ta = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)col;
                asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
                             : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
                               "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
                               "=r"(v[14]), "=r"(v[15])
                             : "r"(ta));
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                if (j < L) {
#pragma unroll
                    for (int q = 0; q < 16; ++q) {
                        const int k = k0 + q;
                        // 32-bit sums: at most 256 entries of magnitude <= L^2 per distance and item
                        if (k > j && k < L) atomicAdd(&sacc[k - j], __float2int_rn(__uint_as_float(v[q])));
                    }
                }
            }
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        }
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        int64_t *rec = ga.rec + (int64_t)r * ga.RL;
        int64_t *D = rec + 3 + (int64_t)axis * (H + 1);
        for (int d = 1 + tid; d <= H; d += GB_THREADS) {
            const long long s2 = (long long)sacc[d] + sacc[L - d];
            sacc[d] = 0;
            sacc[L - d] = 0;
            if (s2) {
                atomicAdd(reinterpret_cast<unsigned long long *>(D + d), (unsigned long long)(-(s2 / 2)));
                if (d == 1) atomicAdd(reinterpret_cast<unsigned long long *>(rec + 2), (unsigned long long)(-(s2 / 2)));
            }
        }
        if (tid == 0 && axis == 2 && un.ra == 0) {
            atomicAdd(reinterpret_cast<unsigned long long *>(rec + 1), (unsigned long long)(2ll * pops[nitem & 1u]));
            pops[nitem & 1u] = 0;  // used again two items on, after the next item's barriers
        }
        g0 += (uint32_t)n;
    }
    if (tid == 0 && !*(volatile int *)&flag) atomicCAS(ga.err, 0, 1);
    if (tid == 0 && mma_pending) atomicExch(ga.err, 2);
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (warp == PW && !mma_pending)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ga.ncols));
}

// Sizes the kernel takes: rows of whole words, distance sums that fit their 32 bits.
bool gram_supported(int L) { return L >= 64 && L <= 2048 && L % 64 == 0; }

// Sizes of the explicit option ISING_CORR_TENSOR.
bool corr_mma_supported(int L) { return L >= 256 && L <= 2048 && L % 128 == 0; }

// What a context or batch class of L >= 512 holds for the measurement: the copies in line order of
// up to 5 replicas (16 where only the x axis has one) at a time fill it.
size_t corr_mma_scratch_bytes(int L, int R)
{
    (void)R;
    return (size_t)2 * L * L * L;
}

template <int PW, int MINB, int READS>
static cudaError_t launch_gram(const GramArgs &ga, int grid, size_t smem, cudaStream_t s, bool pdl)
{
    auto kern = k_gram_bits<PW, MINB, READS>;
    const cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3((unsigned)grid);
    lc.blockDim = dim3(32 * (PW + 2));
    lc.dynamicSmemBytes = smem;
    lc.stream = s;
    cudaLaunchAttribute attr[1] = {pdl_attribute()};
    lc.attrs = attr;
    lc.numAttrs = pdl ? 1 : 0;
    return cudaLaunchKernelEx(&lc, kern, ga);
}

// rec: records initialised to D = N / 2 (r >= 1), M = -N, B = 3 N / 2.  scratch: 2 L^3 bytes for
// the copies in line order, or null (the kernel then reads the packed store: below L = 512, where a word
// is read by one to three units only, for sizes that corr_mma_supported refuses, and where the scratch
// could not be allocated).
cudaError_t launch_corr_mma(const uint32_t *lat, int L, int R, int64_t *rec, uint32_t *scratch, int *err,
                            cudaStream_t s, int64_t *launches, bool pdl, double timeout_s, int inject)
{
    if (!gram_supported(L)) return cudaErrorInvalidValue;
    const Geom g = make_geom(L);
    const bool lines = scratch != nullptr && L >= 512, all3 = g.W % 4 == 0;
    const int per = !lines ? R : (all3 ? 5 : 16);  // replicas per pass: the scratch holds 16 copies
    GramArgs ga{};
    ga.rec = rec;
    ga.RL = 3 + 3 * (int64_t)(L / 2 + 1);
    ga.nw = g.nw;
    ga.L = L;
    ga.W = g.W;
    ga.nsb = (L + 255) / 256;
    ga.nunits = ga.nsb;
    const int nb = (L + 127) / 128;
    for (int bj = 0; bj < nb; ++bj) ga.nunits += ga.nsb - 1 - bj / 2;
    // one stage: 16 KB (one tile), 32 KB (one super-tile) or 48 KB (super-tile and A tile; 32 where the
    // A tile is in tensor memory, which needs whole super-tiles).  Up to
    // L = 128 half of the tensor memory and of the shared memory suffice, so two CTAs share an SM
    // and one's read-back overlaps the other's products.
    const bool small = L <= 128;
    ga.stage_bytes = small ? 16384 : (L <= 256 ? 32768 : 49152);
    ga.nst = L <= 256 ? 6 : 4;
    ga.ncols = small ? 256 : 512;
    ga.scale_col = small ? 128 : 384;
    if (lines && all3) ga.stage_bytes = 32768, ga.nst = 6;  // GR_T
    ga.err = err;
    ga.timeout_ns = (uint64_t)(timeout_s * 1e9);
    const size_t smem = (size_t)ga.nst * ga.stage_bytes + 1024;
    const int slots = device_sms() * (small ? 2 : 1);
    const int nk = (int)((int64_t)L * L / GB_LINES);
    for (int r0 = 0; r0 < R; r0 += per) {
        const int nr = std::min(per, R - r0);
        ga.lat = lat + 2 * (int64_t)r0 * g.nw;
        ga.rec = rec + (int64_t)r0 * ga.RL;
        ga.lines = lines ? scratch : nullptr;
        ga.rep_words = (all3 ? 3 : 1) * 2 * g.nw;
        if (lines) {
            k_lines_x<<<dim3((unsigned)((g.W + 3) / 4), (unsigned)nk, (unsigned)nr), 256, 0, s>>>(ga.lat, g, scratch,
                                                                                                ga.rep_words);
            if (all3)
                k_lines_yz<<<dim3((unsigned)(L / 32), (unsigned)L, (unsigned)(2 * nr)), 256, 0, s>>>(ga.lat, g, scratch,
                                                                                                     ga.rep_words);
        }
        // slices of the lines: the counts whose items take the fewest stages over the CTAs, counting an
        // item's start and read-back as 8 stages, and from L = 512 a stage of the x axis as 1.5 where the
        // kernel transposes it, so that axis is cut finer.  A record of one L = 576 replica takes 227 us
        // that way and 246 with equal slices, of one L = 704 439 and 443; of two L = 320 80 and 69, of one
        // L = 448 89 and 75, of eight L = 256 46 and 44, of six L = 128 14.2 and 13.2.
        ga.nrep = nr;
        const int64_t base = (int64_t)nr * ga.nunits;
        const double wx = lines || L < 512 ? 1.0 : 1.5;
        double best = 1e300;
        for (int sp = 1; sp <= std::min(nk, 64); ++sp) {
            const int sx = std::min(nk, (int)(wx * sp + 0.5));
            const int64_t items = base * (sx + 2 * sp);
            const double tx = wx * ((nk + sx - 1) / sx) + 8.0, ty = (double)((nk + sp - 1) / sp) + 8.0;
            const int64_t rounds = (items + slots - 1) / slots;
            const double cost = (double)rounds * std::max(tx, ty);
            if (cost < best * 0.999) best = cost, ga.split_x = sx, ga.split_yz = sp;
        }
        ga.nitems = (int)(base * (ga.split_x + 2 * ga.split_yz));
        ga.inject = inject && r0 == 0;
        const int grid = std::min(ga.nitems, slots);
        cudaError_t e;
        if (small) e = launch_gram<12, 2, GR_SMALL>(ga, grid, smem, s, pdl);
        else if (lines && all3) e = launch_gram<24, 1, GR_T>(ga, grid, smem, s, pdl);
        else if (all3) e = launch_gram<24, 1, GR_XL>(ga, grid, smem, s, pdl);
        else e = launch_gram<12, 1, GR_ANY>(ga, grid, smem, s, pdl);
        if (e != cudaSuccess) return e;
        if (launches) *launches += !lines ? 1 : (all3 ? 3 : 2);
    }
    return cudaGetLastError();
}

}  // namespace ising
