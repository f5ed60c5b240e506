// sha256_kernels.cu — SHA-256 (FIPS 180-4) on the GPU for page digests.
//
// The digest of a page is SHA-256 over the concatenated SHA-256 digests of its
// consecutive 4096-byte leaves.  A leaf is a serial Merkle-Damgard chain, so
// the natural mapping is one thread per leaf (65 compressions for a 4 KB
// leaf); a second kernel hashes each page's leaf digests with one thread per
// page.  Integer-ALU bound: ~1.7k simple integer ops per 64-byte block.
#include "common.cuh"

namespace kvg {

namespace {

// FIPS 180-4 sec. 4.2.2 round constants and sec. 5.3.3 initial hash value.
__constant__ uint32_t kK[64] = {
    0x428a2f98u, 0x71374491u, 0xb5c0fbcfu, 0xe9b5dba5u, 0x3956c25bu, 0x59f111f1u, 0x923f82a4u,
    0xab1c5ed5u, 0xd807aa98u, 0x12835b01u, 0x243185beu, 0x550c7dc3u, 0x72be5d74u, 0x80deb1feu,
    0x9bdc06a7u, 0xc19bf174u, 0xe49b69c1u, 0xefbe4786u, 0x0fc19dc6u, 0x240ca1ccu, 0x2de92c6fu,
    0x4a7484aau, 0x5cb0a9dcu, 0x76f988dau, 0x983e5152u, 0xa831c66du, 0xb00327c8u, 0xbf597fc7u,
    0xc6e00bf3u, 0xd5a79147u, 0x06ca6351u, 0x14292967u, 0x27b70a85u, 0x2e1b2138u, 0x4d2c6dfcu,
    0x53380d13u, 0x650a7354u, 0x766a0abbu, 0x81c2c92eu, 0x92722c85u, 0xa2bfe8a1u, 0xa81a664bu,
    0xc24b8b70u, 0xc76c51a3u, 0xd192e819u, 0xd6990624u, 0xf40e3585u, 0x106aa070u, 0x19a4c116u,
    0x1e376c08u, 0x2748774cu, 0x34b0bcb5u, 0x391c0cb3u, 0x4ed8aa4au, 0x5b9cca4fu, 0x682e6ff3u,
    0x748f82eeu, 0x78a5636fu, 0x84c87814u, 0x8cc70208u, 0x90befffau, 0xa4506cebu, 0xbef9a3f7u,
    0xc67178f2u};
__constant__ uint32_t kH0[8] = {0x6a09e667u, 0xbb67ae85u, 0x3c6ef372u, 0xa54ff53au,
                                0x510e527fu, 0x9b05688cu, 0x1f83d9abu, 0x5be0cd19u};

__device__ __forceinline__ uint32_t rotr(uint32_t x, int n) { return __funnelshift_r(x, x, n); }

// The integer ALU pipe is this kernel's bottleneck while the FMA pipe idles.
// Additions written as a*one + b and right shifts written as the high word of
// a*2^(32-n) execute as IMAD on the FMA pipe.  `one` is a kernel argument
// (always 1) so the compiler cannot fold the multiply back into an add.
// FMA = false: plain additions and shifts (the compiler fuses them into
// 3-input IADD3 on the ALU pipe) for a serial chain, where the dependency
// chain's latency, not pipe throughput, sets the pace.
template <bool FMA = true>
__device__ __forceinline__ uint32_t fadd(uint32_t a, uint32_t b, uint32_t one) {
    if (!FMA) return a + b;
    uint32_t d;
    asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(one), "r"(b));
    return d;
}
template <int N, bool FMA = true>
__device__ __forceinline__ uint32_t fshr(uint32_t x, uint32_t one) {
    if (!FMA) return x >> N;
    uint32_t d;
    asm("mul.hi.u32 %0, %1, %2;" : "=r"(d) : "r"(x), "r"(one << (32 - N)));
    return d;
}

__device__ __forceinline__ uint32_t bswap(uint32_t x) { return __byte_perm(x, 0, 0x0123); }

// One compression of the 16-word block w (FIPS 180-4 sec. 6.2.2), with the
// message schedule kept as a rolling 16-word window.  Rotations and logic
// stay on the ALU pipe; additions and the schedule's plain shifts go to the
// FMA pipe (fadd/fshr), balancing the two.
// LAT: the additions reassociated for launches of few warps per scheduler,
// where the recurrence's latency decides: e[t+1] is one addition behind
// S1(e[t]) (h + K + W + d and Ch are added up before it), and a[t+1] =
// e[t+1] + (S0 + Maj - d) is one behind e[t+1].  One addition a round more.
template <bool FMA = true, bool LAT = false>
__device__ __forceinline__ void compress(uint32_t st[8], uint32_t w[16], uint32_t one) {
    uint32_t a = st[0], b = st[1], c = st[2], d = st[3], e = st[4], f = st[5], g = st[6], h = st[7];
#pragma unroll
    for (int t = 0; t < 64; ++t) {
        uint32_t wt;
        if (t < 16) {
            wt = w[t];
        } else {
            const uint32_t w15 = w[(t - 15) & 15], w2 = w[(t - 2) & 15];
            const uint32_t s0 = rotr(w15, 7) ^ rotr(w15, 18) ^ fshr<3, FMA>(w15, one);
            const uint32_t s1 = rotr(w2, 17) ^ rotr(w2, 19) ^ fshr<10, FMA>(w2, one);
            wt = w[t & 15] = fadd<FMA>(fadd<FMA>(w[t & 15], s0, one), fadd<FMA>(w[(t - 7) & 15], s1, one), one);
        }
        const uint32_t S1 = rotr(e, 6) ^ rotr(e, 11) ^ rotr(e, 25);
        const uint32_t ch = (e & f) ^ (~e & g);
        if (LAT) {
            const uint32_t y = fadd<FMA>(fadd<FMA>(fadd<FMA>(wt, kK[t], one), h, one), d, one);
            const uint32_t ne = fadd<FMA>(fadd<FMA>(y, ch, one), S1, one);
            const uint32_t S0 = rotr(a, 2) ^ rotr(a, 13) ^ rotr(a, 22);
            const uint32_t maj = (a & b) ^ (a & c) ^ (b & c);
            uint32_t md;  // Maj - d
            asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(md) : "r"(d), "r"(0u - one), "r"(maj));
            h = g;
            g = f;
            f = e;
            e = ne;
            d = c;
            c = b;
            b = a;
            a = fadd<FMA>(ne, fadd<FMA>(S0, md, one), one);
            continue;
        }
        const uint32_t T1 = fadd<FMA>(fadd<FMA>(h, S1, one), fadd<FMA>(fadd<FMA>(ch, kK[t], one), wt, one), one);
        const uint32_t S0 = rotr(a, 2) ^ rotr(a, 13) ^ rotr(a, 22);
        const uint32_t maj = (a & b) ^ (a & c) ^ (b & c);
        h = g;
        g = f;
        f = e;
        e = fadd<FMA>(d, T1, one);
        d = c;
        c = b;
        b = a;
        a = fadd<FMA>(T1, fadd<FMA>(S0, maj, one), one);
    }
    st[0] += a;
    st[1] += b;
    st[2] += c;
    st[3] += d;
    st[4] += e;
    st[5] += f;
    st[6] += g;
    st[7] += h;
}

__device__ __forceinline__ void init_state(uint32_t st[8]) {
#pragma unroll
    for (int i = 0; i < 8; ++i) st[i] = kH0[i];
}

// Final block(s) for a message whose last `rem` (< 64) bytes start at `tail`
// and whose total length is `total_bytes`.
__device__ void finish(uint32_t st[8], const uint8_t *tail, int rem, uint64_t total_bytes, uint32_t one) {
    uint32_t w[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) w[i] = 0;
    for (int k = 0; k < rem; ++k) w[k >> 2] |= (uint32_t)tail[k] << (24 - 8 * (k & 3));
    w[rem >> 2] |= 0x80u << (24 - 8 * (rem & 3));
    const uint64_t bits = total_bytes * 8ull;
    if (rem < 56) {
        w[14] = (uint32_t)(bits >> 32);
        w[15] = (uint32_t)bits;
        compress(st, w, one);
    } else {
        compress(st, w, one);
#pragma unroll
        for (int i = 0; i < 16; ++i) w[i] = 0;
        w[14] = (uint32_t)(bits >> 32);
        w[15] = (uint32_t)bits;
        compress(st, w, one);
    }
}

__device__ __forceinline__ const uint8_t *page_addr(const PageSource &s, int64_t p) {
    if (!s.pid) return s.base + (uint64_t)p * s.page_bytes;
    const int64_t plane = p / s.npb;
    const int64_t j = p - plane * s.npb;
    return s.base + ((uint64_t)plane * s.plane_pages + (uint64_t)s.pid[j]) * s.page_bytes;
}

// 16-byte asynchronous copy global -> this thread's shared memory (LDGSTS,
// L1 bypassed); completion is tracked by the thread's cp.async groups.
__device__ __forceinline__ void cp_async16(void *smem_dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_addr(smem_dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_async_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory"); }

// SHA-256 of one leaf that is also copied to `copy_to`, from the same
// registers that are hashed, so the bytes written are exactly the bytes whose
// digest is checked.  The leaf's next R 64-byte blocks are in flight through
// a ring of this thread's shared memory (ring: R x 64 contiguous bytes), not
// held in registers, so their latency (long when other kernels keep HBM
// busy) hides behind the compressions without costing registers.  (A layout
// with the 32 lanes' vectors side by side, free of bank conflicts, measured
// slower in the 12b step: 6.05 against 5.94 ms.)
template <int R>
__device__ __forceinline__ void hash_leaf_ring(const uint8_t *leaf, uint64_t len, uint8_t *copy_to, uint32_t st[8],
                                               uint32_t one, uint4 *ring) {
    const uint4 *v = reinterpret_cast<const uint4 *>(leaf);
    uint4 *o = reinterpret_cast<uint4 *>(copy_to);
    init_state(st);
    const int nfull = (int)(len >> 6);
#pragma unroll
    for (int b = 0; b < R; ++b) {
        if (b < nfull)
#pragma unroll
            for (int q = 0; q < 4; ++q) cp_async16(ring + 4 * b + q, v + 4 * b + q);
        cp_async_commit();  // one group per block, empty or not, so the count stays uniform
    }
    for (int blk = 0; blk < nfull; ++blk) {
        cp_async_wait<R - 1>();  // block blk has landed
        const int slot = blk % R;
        uint32_t w[16];
        uint4 x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) x[q] = ring[4 * slot + q];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            w[4 * q + 0] = bswap(x[q].x);
            w[4 * q + 1] = bswap(x[q].y);
            w[4 * q + 2] = bswap(x[q].z);
            w[4 * q + 3] = bswap(x[q].w);
        }
        // the slot is free once its words are in registers: refill it
        if (blk + R < nfull)
#pragma unroll
            for (int q = 0; q < 4; ++q) cp_async16(ring + 4 * slot + q, v + 4 * (blk + R) + q);
        cp_async_commit();
#pragma unroll
        for (int q = 0; q < 4; ++q) __stcs(o + 4 * blk + q, x[q]);
        compress(st, w, one);
    }
    cp_async_wait<0>();
    const int rem = (int)(len & 63);
    if (rem == 0) {
        uint32_t w[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) w[q] = 0;
        w[0] = 0x80000000u;
        const uint64_t bits = len * 8ull;
        w[14] = (uint32_t)(bits >> 32);
        w[15] = (uint32_t)bits;
        compress(st, w, one);
    } else {
        for (int q = 0; q < rem / 16; ++q) o[4 * nfull + q] = v[4 * nfull + q];
        finish(st, leaf + (len & ~63ull), rem, len, one);
    }
}

// SHA-256 of one leaf of `len` bytes (16-byte aligned).  With COPY the leaf
// is also written to `copy_to`, from the same registers that are hashed, so
// the bytes written are exactly the bytes whose digest is checked.
template <bool COPY, bool LAT = false>
__device__ __forceinline__ void hash_leaf(const uint8_t *leaf, uint64_t len, uint8_t *copy_to, uint32_t st[8],
                                          uint32_t one) {
    const uint4 *v = reinterpret_cast<const uint4 *>(leaf);
    uint4 *o = reinterpret_cast<uint4 *>(copy_to);
    init_state(st);
    const int nfull = (int)(len >> 6);
    // The next two 64-byte blocks are in flight while the current one is
    // compressed, so their memory latency (long when other kernels keep HBM
    // busy) hides behind ~3.4k ALU ops.
    uint4 n1[4], n2[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        if (nfull > 0) n1[q] = v[q];
        if (nfull > 1) n2[q] = v[4 + q];
    }
    for (int blk = 0; blk < nfull; ++blk) {
        uint32_t w[16];
        uint4 x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            x[q] = n1[q];
            n1[q] = n2[q];
        }
        if (blk + 2 < nfull) {
#pragma unroll
            for (int q = 0; q < 4; ++q) n2[q] = v[4 * (blk + 2) + q];
        }
        if (COPY) {
#pragma unroll
            for (int q = 0; q < 4; ++q) __stcs(o + 4 * blk + q, x[q]);
        }
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            w[4 * q + 0] = bswap(x[q].x);
            w[4 * q + 1] = bswap(x[q].y);
            w[4 * q + 2] = bswap(x[q].z);
            w[4 * q + 3] = bswap(x[q].w);
        }
        compress<true, LAT>(st, w, one);
    }
    const int rem = (int)(len & 63);
    if (rem == 0) {
        uint32_t w[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) w[q] = 0;
        w[0] = 0x80000000u;
        const uint64_t bits = len * 8ull;
        w[14] = (uint32_t)(bits >> 32);
        w[15] = (uint32_t)bits;
        compress<true, LAT>(st, w, one);
    } else {
        if (COPY)
            for (int q = 0; q < rem / 16; ++q) o[4 * nfull + q] = v[4 * nfull + q];
        finish(st, leaf + (len & ~63ull), rem, len, one);
    }
}

__device__ __forceinline__ void store_state(uint32_t *out, const uint32_t st[8]) {
    uint4 *o = reinterpret_cast<uint4 *>(out);
    o[0] = make_uint4(st[0], st[1], st[2], st[3]);
    o[1] = make_uint4(st[4], st[5], st[6], st[7]);
}

// ---- two-warp form, for launches too small to fill the GPU ---------------
// When there are few chains, each one's latency decides.  Two warps of a
// 64-thread CTA share the work: one loads the message, expands the schedule
// and leaves K[t] + W[t] in shared memory, the other runs the rounds.
//
// A compression's 64 rounds are one recurrence with two halves: e[t+1] needs
// a[t-3], four rounds old, and a[t+1] = (e[t+1] - a[t-3]) + S0(a[t]) + maj.  So
// a chain takes two lanes: lane c (c < 16) runs the e half at round t while
// lane c + 16 runs the a half two rounds behind, and one shuffle per round
// (each lane's new word to its partner, used two rounds later, so its latency
// is hidden) carries both couplings.  Both halves are the same instructions
// with per-lane rotation amounts: new = rotr(x, r1) ^ rotr(x, r2) ^ rotr(x, r3)
// + choose + in, where maj(a, b, c) is b where a and b agree and c elsewhere,
// i.e. a choose whose selector is ~(a ^ b).  What bounds it is the latency of
// rotation, xor and addition, one after the other, once a round; a lane that
// runs both halves adds twice their ALU work to it.  A lone chain takes 0.74
// us per 64-byte block against 0.84 with both halves in one lane (and 1.46 in
// one warp), the digests of 64 leaves 70 us against 77.  The loading warp's
// half-warps take one block each, so a hand-over is a pair of blocks; the a
// lanes read zeros for their K + W.
//
// The wide form runs both halves in one lane, 32 chains per CTA, a block per
// hand-over: a leaf launch of 33 to 64 leaves per SM takes it, where four CTAs
// of the other would put a loading warp beside every rounds' warp on its
// scheduler (64 leaves per SM: 76 us wide, 92 with two lanes, 109 in one warp).
//
// Two buffers change hands through named barriers: 1 + b (buffer b full: the
// loading warp arrives, the rounds' warp waits) and 3 + b (buffer b free
// again: the rounds' warp arrives, the loading warp waits).  Both warps run
// the same number of hand-overs, with every lane taking part (lanes past the
// last chain hash zeros and store nothing), so every arrival meets its wait.
constexpr int kSplitChains = 16;
constexpr int kWideChains = 32;

struct __align__(16) SplitShared {
    // [buffer][block of the pair, or upper half of the wide form's chains]
    // [t / 4][chain], 4 consecutive t each
    uint4 kw[2][2][16][kSplitChains];
    uint4 zero[16][kSplitChains];      // what the a lanes read
    int consumer;                      // which of the two warps runs the rounds
};

__device__ __forceinline__ void bar_sync_pair(int id) { asm volatile("bar.sync %0, 64;" ::"r"(id) : "memory"); }
__device__ __forceinline__ void bar_arrive_pair(int id) { asm volatile("bar.arrive %0, 64;" ::"r"(id) : "memory"); }

// The loading warp: the message schedule of block w plus the round constants, into
// column c of kw[16][kSplitChains].  Additions and plain shifts go to the FMA
// pipe (fadd, fshr), which leaves the ALU pipe to a rounds' warp on the same
// scheduler.
__device__ __forceinline__ void split_expand(uint4 (*kw)[kSplitChains], uint32_t w[16], int c, uint32_t one) {
#pragma unroll
    for (int t4 = 0; t4 < 16; ++t4) {
        uint32_t v[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
            const int t = 4 * t4 + i;
            uint32_t wt;
            if (t < 16) {
                wt = w[t];
            } else {
                const uint32_t w15 = w[(t - 15) & 15], w2 = w[(t - 2) & 15];
                const uint32_t s0 = rotr(w15, 7) ^ rotr(w15, 18) ^ fshr<3>(w15, one);
                const uint32_t s1 = rotr(w2, 17) ^ rotr(w2, 19) ^ fshr<10>(w2, one);
                wt = w[t & 15] = fadd(fadd(fadd(w[t & 15], w[(t - 7) & 15], one), s0, one), s1, one);
            }
            v[i] = fadd(wt, kK[t], one);
        }
        kw[t4][c] = make_uint4(v[0], v[1], v[2], v[3]);
    }
}

// The rounds' warp, per lane: which half of the recurrence it runs.
struct SplitRole {
    int r1, r2, r3;   // rotations of its sum function
    uint32_t sign;    // 1 (e: + h) or -1 (a: - d), as a factor
    uint32_t agree;   // 0 (choose by x) or ~0 (by ~(x ^ y))
    bool a;
};
__device__ __forceinline__ SplitRole split_role(int lane) {
    const bool a = lane >= kSplitChains;
    return SplitRole{a ? 2 : 6, a ? 13 : 11, a ? 22 : 25, a ? 0xffffffffu : 1u, a ? 0xffffffffu : 0u, a};
}

// The rounds' warp: the 64 rounds of one block (FIPS 180-4 sec. 6.2.2 step 3) and the
// feed-forward.  st is the lane's half of the state: e, f, g, h or a, b, c, d.
// At step s the e lanes run round s and the a lanes round s - 2: in the
// first two steps the a lanes only bring b and a into their window (which
// starts as c, d), and after step 63 the e lanes' steps are ignored.
__device__ __forceinline__ void split_rounds(uint32_t st[4], const uint4 *kw, const SplitRole &ro, uint32_t one) {
    uint32_t p1 = ro.a ? st[2] : st[0], p2 = ro.a ? st[3] : st[1], p3 = st[2], p4 = st[3];
    // the partner's words of two steps ago; before step 0: the e lanes get d, then c
    uint32_t sh0 = __shfl_xor_sync(0xffffffffu, st[3], kSplitChains);
    uint32_t sh1 = __shfl_xor_sync(0xffffffffu, st[2], kSplitChains);
    uint32_t e1 = 0, e2 = 0, e3 = 0, e4 = 0;
    uint4 k4 = make_uint4(0, 0, 0, 0);
#pragma unroll
    for (int s = 0; s < 66; ++s) {
        if (s < 64 && (s & 3) == 0) k4 = kw[(s >> 2) * kSplitChains];
        const uint32_t k = s >= 64 ? 0u : (s & 3) == 0 ? k4.x : (s & 3) == 1 ? k4.y : (s & 3) == 2 ? k4.z : k4.w;
        uint32_t q;  // h + K[t] + W[t], or -d
        asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(q) : "r"(p4), "r"(ro.sign), "r"(k));
        const uint32_t in = fadd(sh0, q, one);
        const uint32_t S = __funnelshift_r(p1, p1, ro.r1) ^ __funnelshift_r(p1, p1, ro.r2) ^
                           __funnelshift_r(p1, p1, ro.r3);
        const uint32_t sel = p1 ^ (~p2 & ro.agree);
        const uint32_t ch = (sel & p2) ^ (~sel & p3);
        uint32_t n = S + ch + in;
        if (s == 0) n = ro.a ? st[1] : n;
        if (s == 1) n = ro.a ? st[0] : n;
        sh0 = sh1;
        if (s < 64) sh1 = __shfl_xor_sync(0xffffffffu, n, kSplitChains);
        p4 = p3;
        p3 = p2;
        p2 = p1;
        p1 = n;
        if (s == 63) {
            e1 = p1;
            e2 = p2;
            e3 = p3;
            e4 = p4;
        }
    }
    st[0] += ro.a ? p1 : e1;
    st[1] += ro.a ? p2 : e2;
    st[2] += ro.a ? p3 : e3;
    st[3] += ro.a ? p4 : e4;
}

// Both warps, before their loops: the zeros of the a lanes, and which warp
// does what (true: this one loads and expands).  A CTA's two warps sit on
// neighbouring schedulers, so with warp 0 always running the rounds, four
// CTAs on an SM would put their rounds on two of the four schedulers (105
// instead of 90 us at 64 leaves per SM); every other pair of warp slots swaps
// the roles instead.  The slot number is only read here, by one thread.
__device__ __forceinline__ bool split_begin(SplitShared &sm) {
    for (int i = threadIdx.x; i < 16 * kSplitChains; i += 64) (&sm.zero[0][0])[i] = make_uint4(0, 0, 0, 0);
    if (threadIdx.x == 0) {
        uint32_t slot;
        asm volatile("mov.u32 %0, %%warpid;" : "=r"(slot));
        sm.consumer = (int)((slot >> 2) & 1);
    }
    __syncthreads();
    after_previous();
    return (int)(threadIdx.x >> 5) != sm.consumer;
}

// The rounds' warp over a chain of n_blocks blocks: its half of the state from
// H0 (from: a stored state's words) to the digest.
__device__ __forceinline__ void split_consume(uint32_t st[4], const SplitShared &sm, int n_blocks, int lane,
                                              uint32_t one, const uint32_t *from = nullptr) {
    const SplitRole ro = split_role(lane);
    const int c = lane & (kSplitChains - 1);
#pragma unroll
    for (int i = 0; i < 4; ++i) st[i] = from ? from[i + (ro.a ? 0 : 4)] : kH0[i + (ro.a ? 0 : 4)];
    const int n_pairs = (n_blocks + 1) >> 1;
    for (int k = 0; k < n_pairs; ++k) {
        const int buf = k & 1;
        bar_sync_pair(1 + buf);
#pragma unroll 1
        for (int h = 0; h < 2 && 2 * k + h < n_blocks; ++h) {
            if (2 * k + h == n_blocks - 1) let_next_start();
            split_rounds(st, ro.a ? &sm.zero[0][c] : &sm.kw[buf][h][0][c], ro, one);
        }
        if (k + 2 < n_pairs) bar_arrive_pair(3 + buf);
    }
}

// The wide form's rounds of one block: both halves of the state in one lane.
// The additions off the last step go to the FMA pipe (fadd): e[t+1] is one
// addition behind S1(e[t]) and a[t+1] = e[t+1] + S0 + (maj - d) one behind that.
__device__ __forceinline__ void wide_rounds(uint32_t st[8], const uint4 *kw, uint32_t one) {
    uint32_t a = st[0], b = st[1], c = st[2], d = st[3], e = st[4], f = st[5], g = st[6], h = st[7];
    uint4 k4 = make_uint4(0, 0, 0, 0);
#pragma unroll
    for (int t = 0; t < 64; ++t) {
        if ((t & 3) == 0) k4 = kw[(t >> 2) * kSplitChains];
        const uint32_t k = (t & 3) == 0 ? k4.x : (t & 3) == 1 ? k4.y : (t & 3) == 2 ? k4.z : k4.w;
        const uint32_t S1 = rotr(e, 6) ^ rotr(e, 11) ^ rotr(e, 25);
        const uint32_t ch = (e & f) ^ (~e & g);
        const uint32_t S0 = rotr(a, 2) ^ rotr(a, 13) ^ rotr(a, 22);
        const uint32_t maj = (a & b) ^ (a & c) ^ (b & c);
        const uint32_t y = fadd(fadd(fadd(h, k, one), d, one), ch, one);
        uint32_t md;  // maj - d
        asm("mad.lo.u32 %0, %1, %2, %3;" : "=r"(md) : "r"(d), "r"(0u - one), "r"(maj));
        const uint32_t ne = S1 + y;
        h = g;
        g = f;
        f = e;
        e = ne;
        d = c;
        c = b;
        b = a;
        a = ne + S0 + md;
    }
    st[0] += a;
    st[1] += b;
    st[2] += c;
    st[3] += d;
    st[4] += e;
    st[5] += f;
    st[6] += g;
    st[7] += h;
}

// The rounds' warp of the wide form over a chain of n_blocks blocks.
__device__ __forceinline__ void wide_consume(uint32_t st[8], const SplitShared &sm, int n_blocks, int lane,
                                             uint32_t one) {
    init_state(st);
    for (int k = 0; k < n_blocks; ++k) {
        const int buf = k & 1;
        bar_sync_pair(1 + buf);
        if (k == n_blocks - 1) let_next_start();
        wide_rounds(st, &sm.kw[buf][lane / kSplitChains][0][lane & (kSplitChains - 1)], one);
        if (k + 2 < n_blocks) bar_arrive_pair(3 + buf);
    }
}

// A lane of the loading warp hands over its block of pair (wide form: its
// chain's block) k, 16 words in w, through buffer k & 1.
__device__ __forceinline__ void split_hand_over(SplitShared &sm, uint32_t w[16], int k, int lane, uint32_t one) {
    const int buf = k & 1;
    if (k >= 2) bar_sync_pair(3 + buf);
    split_expand(sm.kw[buf][lane / kSplitChains], w, lane & (kSplitChains - 1), one);
    __threadfence_block();
    bar_arrive_pair(1 + buf);
}

// The padding block of a message of `bytes` bytes (a multiple of 64).
__device__ __forceinline__ void padding_block(uint32_t w[16], uint64_t bytes) {
#pragma unroll
    for (int q = 0; q < 16; ++q) w[q] = 0;
    w[0] = 0x80000000u;
    const uint64_t bits = bytes * 8ull;
    w[14] = (uint32_t)(bits >> 32);
    w[15] = (uint32_t)bits;
}

// The loading warp over a whole 4 KiB leaf at v (nullptr: zeros), also written
// to o when COPY (the bytes written are the bytes hashed): 32 pairs of data
// blocks (wide form: 64 blocks), the next two in flight, then the padding
// block.
template <bool COPY, bool WIDE>
__device__ __forceinline__ void split_produce_leaf(SplitShared &sm, const uint4 *v, uint4 *o, int lane,
                                                   uint32_t one) {
    constexpr int kStep = WIDE ? 4 : 8;  // vectors of the leaf per hand-over
    constexpr int kHandOvers = (int)(kLeafBytes / 16) / kStep;
    if (!WIDE && v) v += 4 * (lane / kSplitChains);
    if (!WIDE && COPY && o) o += 4 * (lane / kSplitChains);
    uint4 n1[4], n2[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) {
        n1[q] = v ? v[q] : make_uint4(0, 0, 0, 0);
        n2[q] = v ? v[kStep + q] : make_uint4(0, 0, 0, 0);
    }
    for (int k = 0; k < kHandOvers; ++k) {
        uint4 x[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            x[q] = n1[q];
            n1[q] = n2[q];
        }
        if (v && k + 2 < kHandOvers) {
#pragma unroll
            for (int q = 0; q < 4; ++q) n2[q] = v[kStep * (k + 2) + q];
        }
        if (COPY && o) {
#pragma unroll
            for (int q = 0; q < 4; ++q) __stcs(o + kStep * k + q, x[q]);
        }
        uint32_t w[16];
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            w[4 * q + 0] = bswap(x[q].x);
            w[4 * q + 1] = bswap(x[q].y);
            w[4 * q + 2] = bswap(x[q].z);
            w[4 * q + 3] = bswap(x[q].w);
        }
        split_hand_over(sm, w, k, lane, one);
    }
    uint32_t w[16];
    padding_block(w, kLeafBytes);
    split_hand_over(sm, w, kHandOvers, lane, one);
}

constexpr int kSplitLeafBlocks = (int)(kLeafBytes / 64) + 1;

// The rounds' warp over whole 4 KiB leaves: the chain's digest to out (null:
// nothing; zero: zeros instead).
template <bool WIDE>
__device__ __forceinline__ void split_consume_leaf(SplitShared &sm, uint32_t *out, bool zero, int lane, uint32_t one) {
    if (WIDE) {
        uint32_t st[8];
        wide_consume(st, sm, kSplitLeafBlocks, lane, one);
        if (!out) return;
#pragma unroll
        for (int w = 0; w < 8; ++w) st[w] = zero ? 0u : st[w];
        store_state(out, st);
    } else {
        uint32_t st[4];  // words 0-3 (a lanes) or 4-7
        split_consume(st, sm, kSplitLeafBlocks, lane, one);
        if (!out) return;
        reinterpret_cast<uint4 *>(out)[lane >= kSplitChains ? 0 : 1] =
            zero ? make_uint4(0, 0, 0, 0) : make_uint4(st[0], st[1], st[2], st[3]);
    }
}

// The chain of a lane of either warp, within the CTA.
template <bool WIDE>
__device__ __forceinline__ int64_t split_chain(int lane) {
    return WIDE ? (int64_t)blockIdx.x * kWideChains + lane
                : (int64_t)blockIdx.x * kSplitChains + (lane & (kSplitChains - 1));
}

// The whole state in an e lane of the rounds' warp (all lanes take part).
__device__ __forceinline__ void split_whole_state(uint32_t full[8], const uint32_t st[4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        full[i] = __shfl_xor_sync(0xffffffffu, st[i], kSplitChains);
        full[4 + i] = st[i];
    }
}

// graft_verify_kernel's work in the two-warp form, for pages made of whole
// 4 KiB leaves and launches of a few such CTAs per SM.
template <bool WIDE>
__global__ void __launch_bounds__(64) graft_verify_split_kernel(const GraftParams p, int64_t leaves_per_page,
                                                                uint32_t *out, uint32_t one) {
    __shared__ SplitShared sm;
    const bool produce = split_begin(sm);
    graft_metadata(p);
    const int lane = threadIdx.x & 31;
    const uint64_t page_bytes = p.page_bytes;
    const int64_t n_leaves = (int64_t)p.n_layers * 2 * p.npb * leaves_per_page;
    const int64_t idx = split_chain<WIDE>(lane);
    const bool valid = idx < n_leaves;
    const int64_t page_u = idx / leaves_per_page;
    const int64_t i = idx - page_u * leaves_per_page;
    const int64_t lkv = page_u / p.npb;
    const int64_t jj = page_u - lkv * p.npb;
    const int64_t block_page = lkv * p.block_pages + p.page_base + jj;
    if (produce) {
        const uint64_t off = (uint64_t)i * kLeafBytes;
        const uint4 *v = valid ? reinterpret_cast<const uint4 *>(p.src + (uint64_t)block_page * page_bytes + off)
                               : nullptr;
        uint4 *o = valid ? reinterpret_cast<uint4 *>(p.pool + ((uint64_t)lkv * p.pool_pages +
                                                               (uint64_t)p.pids.pid[jj]) * page_bytes + off)
                         : nullptr;
        split_produce_leaf<true, WIDE>(sm, v, o, lane, one);
    } else {
        split_consume_leaf<WIDE>(sm, valid ? out + (block_page * leaves_per_page + i) * 8 : nullptr, false, lane, one);
    }
}

// sha256_leaves_kernel's work in the two-warp form (whole 4 KiB leaves).
template <bool WIDE>
__global__ void __launch_bounds__(64) sha256_leaves_split_kernel(const PageSource src, int64_t n_pages,
                                                                 int64_t leaves_per_page,
                                                                 uint32_t *out, uint32_t one) {
    __shared__ SplitShared sm;
    const bool produce = split_begin(sm);
    const int lane = threadIdx.x & 31;
    const int64_t idx = split_chain<WIDE>(lane);
    const bool valid = idx < n_pages * leaves_per_page;
    const int64_t p = idx / leaves_per_page;
    const int64_t i = idx - p * leaves_per_page;
    bool in_range = valid;
    if (valid && src.pid) {  // page ids come from a device page table: never read outside the pool
        const int32_t pid = src.pid[p - (p / src.npb) * src.npb];
        in_range = pid >= 0 && pid < src.plane_pages;
    }
    if (produce) {
        const uint4 *v = in_range ? reinterpret_cast<const uint4 *>(page_addr(src, p) + (uint64_t)i * kLeafBytes)
                                  : nullptr;
        split_produce_leaf<false, WIDE>(sm, v, nullptr, lane, one);
    } else {
        int64_t po = p;
        if (src.pid && src.out_plane_stride) {
            const int64_t plane = p / src.npb;
            po = plane * src.out_plane_stride + src.out_j0 + (p - plane * src.npb);
        }
        // a page id out of range has no digest: zeros, reported as a mismatch
        split_consume_leaf<WIDE>(sm, valid ? out + (po * leaves_per_page + i) * 8 : nullptr, !in_range, lane, one);
    }
}

template <bool LAT>
__global__ void __launch_bounds__(128) sha256_leaves_kernel(const PageSource src, int64_t n_pages,
                                                            int64_t leaves_per_page,
                                                            uint32_t *out, uint32_t one) {
    after_previous();
    const int64_t n_leaves = n_pages * leaves_per_page;
    for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < n_leaves;
         idx += (int64_t)gridDim.x * blockDim.x) {
        const int64_t p = idx / leaves_per_page;
        const int64_t i = idx - p * leaves_per_page;
        uint64_t len = src.page_bytes - (uint64_t)i * kLeafBytes;
        if (len > kLeafBytes) len = kLeafBytes;
        uint32_t st[8];
        bool in_range = true;
        if (src.pid) {  // page ids come from a device page table: never read outside the pool
            const int32_t pid = src.pid[p - (p / src.npb) * src.npb];
            in_range = pid >= 0 && pid < src.plane_pages;
        }
        if (in_range) {
            hash_leaf<false, LAT>(page_addr(src, p) + (uint64_t)i * kLeafBytes, len, nullptr, st, one);
        } else {
#pragma unroll
            for (int w = 0; w < 8; ++w) st[w] = 0u;  // no digest of any page: reported as a mismatch
        }
        int64_t po = p;
        if (src.pid && src.out_plane_stride) {
            const int64_t plane = p / src.npb;
            po = plane * src.out_plane_stride + src.out_j0 + (p - plane * src.npb);
        }
        store_state(out + (po * leaves_per_page + i) * 8, st);
    }
}

// graft_verify_kernel with each thread keeping its leaf's next
// kGraftVerifyRing blocks in flight through its own slots of shared memory
// instead of two blocks in registers; the registers that frees let five CTAs
// of 128 threads stay resident per SM (96 registers).  Used for launches of
// at least one full wave of it (five CTAs on every SM): beside a concurrent
// append the 12b step's window shortens (step 5.94 against 6.01 ms; alone
// the same 3.12 ms; rings of two or four blocks, or six CTAs at 80
// registers, measured slower in the step).  For smaller launches each leaf's
// chain latency decides: the register form is faster there (the tiny
// verified graft 0.099 against 0.133 ms), and the two-warp form faster still
// for launches of up to 64 leaves per SM (0.057 ms).
constexpr int kGraftVerifyRing = 3;
__global__ void __launch_bounds__(128, 5) graft_verify_ring_kernel(const GraftParams p, int64_t leaves_per_page,
                                                                   uint32_t *out, uint32_t one) {
    after_previous();
    constexpr int R = kGraftVerifyRing;
    extern __shared__ __align__(16) uint4 ring_mem[];
    graft_metadata(p);
    const uint64_t page_bytes = p.page_bytes;
    const int64_t n_leaves = (int64_t)p.n_layers * 2 * p.npb * leaves_per_page;
    uint4 *ring = ring_mem + threadIdx.x * 4 * R;
    for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < n_leaves;
         idx += (int64_t)gridDim.x * blockDim.x) {
        const int64_t page_u = idx / leaves_per_page;
        const int64_t i = idx - page_u * leaves_per_page;
        const int64_t lkv = page_u / p.npb;
        const int64_t jj = page_u - lkv * p.npb;
        const uint64_t off = (uint64_t)i * kLeafBytes;
        uint64_t len = page_bytes - off;
        if (len > kLeafBytes) len = kLeafBytes;
        const int64_t block_page = lkv * p.block_pages + p.page_base + jj;
        const uint8_t *src = p.src + (uint64_t)block_page * page_bytes + off;
        uint8_t *dst = p.pool + ((uint64_t)lkv * p.pool_pages + (uint64_t)p.pids.pid[jj]) * page_bytes + off;
        uint32_t st[8];
        hash_leaf_ring<R>(src, len, dst, st, one, ring);
        store_state(out + (block_page * leaves_per_page + i) * 8, st);
    }
}

// Own-position graft with the verification folded into the copy: one thread
// per 4 KiB leaf reads it from the block once, writes it to its cache page and
// hashes it (leaf order of a page digest, Sec. 3.2's integrity check).
__global__ void __launch_bounds__(128) graft_verify_kernel(const GraftParams p, int64_t leaves_per_page,
                                                           uint32_t *out, uint32_t one) {
    after_previous();
    graft_metadata(p);
    const uint64_t page_bytes = p.page_bytes;
    const int64_t n_leaves = (int64_t)p.n_layers * 2 * p.npb * leaves_per_page;
    for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < n_leaves;
         idx += (int64_t)gridDim.x * blockDim.x) {
        const int64_t page_u = idx / leaves_per_page;
        const int64_t i = idx - page_u * leaves_per_page;
        const int64_t lkv = page_u / p.npb;
        const int64_t jj = page_u - lkv * p.npb;
        const uint64_t off = (uint64_t)i * kLeafBytes;
        uint64_t len = page_bytes - off;
        if (len > kLeafBytes) len = kLeafBytes;
        const int64_t block_page = lkv * p.block_pages + p.page_base + jj;
        const uint8_t *src = p.src + (uint64_t)block_page * page_bytes + off;
        uint8_t *dst = p.pool + ((uint64_t)lkv * p.pool_pages + (uint64_t)p.pids.pid[jj]) * page_bytes + off;
        uint32_t st[8];
        hash_leaf<true>(src, len, dst, st, one);
        store_state(out + (block_page * leaves_per_page + i) * 8, st);
    }
}

// ---- a batch of grafts, verified ------------------------------------------
// The leaves of a batch's jobs in one launch, so that a batch of short blocks
// fills the GPU like one long block does: a leaf per thread, leaf fastest,
// then job, then plane (a block's pages follow one another in a plane).  COPY:
// every page is copied and hashed in one pass (the key pages of re-based
// grafts too: the rotating copy that follows overwrites them; the hashing is
// what the launch waits for, so writing them twice costs nothing).  Otherwise
// the pages are in the cache already and are hashed there, re-based grafts' in
// the store.
struct BatchLeaf {
    const uint8_t *src;
    uint8_t *dst;
    uint64_t len;
};

template <bool COPY>
__device__ __forceinline__ BatchLeaf batch_leaf(const GraftBatchParams &p, int64_t idx, int64_t m) {
    const int64_t page = idx / m;
    const int64_t lkv = page / p.slice_jobs;
    const int64_t jb = page - lkv * p.slice_jobs;
    const uint64_t off = (uint64_t)(idx - page * m) * kLeafBytes;
    const GraftJob job = p.jobs[p.job0 + jb];
    BatchLeaf r;
    r.len = p.page_bytes - off;
    if (r.len > kLeafBytes) r.len = kLeafBytes;
    r.src = job.src + (uint64_t)lkv * job.block_pages * p.page_bytes + off;
    r.dst = p.pool + ((uint64_t)lkv * p.pool_pages + (uint64_t)job.pid) * p.page_bytes + off;
    if (!COPY && p.metas[job.meta].trig < 0) r.src = r.dst;
    return r;
}

// graft_verify_ring_kernel for a batch (the same launch sizes).
__global__ void __launch_bounds__(128, 5) graft_batch_verify_ring_kernel(const GraftBatchParams p,
                                                                         int64_t leaves_per_page,
                                                                         uint32_t *out, uint32_t one) {
    after_previous();
    constexpr int R = kGraftVerifyRing;
    extern __shared__ __align__(16) uint4 ring_mem[];
    if (p.write_meta) batch_metadata(p);
    const int64_t n_leaves = p.slice_jobs * p.n_layers * 2 * leaves_per_page;
    uint4 *ring = ring_mem + threadIdx.x * 4 * R;
    // (a loop, though the grid has a thread for every leaf: straight-line, the
    // compiler's schedule of the compressions ran 13% slower, 4.69 against 4.08 ms
    // for 1.06 million leaves)
    for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < n_leaves;
         idx += (int64_t)gridDim.x * blockDim.x) {
        const BatchLeaf l = batch_leaf<true>(p, idx, leaves_per_page);
        uint32_t st[8];
        hash_leaf_ring<R>(l.src, l.len, l.dst, st, one, ring);
        store_state(out + idx * 8, st);
    }
}

// graft_verify_kernel for a batch.
template <bool COPY>
__global__ void __launch_bounds__(128) graft_batch_verify_kernel(const GraftBatchParams p, int64_t leaves_per_page,
                                                                 uint32_t *out, uint32_t one) {
    after_previous();
    if (p.write_meta) batch_metadata(p);
    const int64_t n_leaves = p.slice_jobs * p.n_layers * 2 * leaves_per_page;
    for (int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; idx < n_leaves;
         idx += (int64_t)gridDim.x * blockDim.x) {
        const BatchLeaf l = batch_leaf<COPY>(p, idx, leaves_per_page);
        uint32_t st[8];
        hash_leaf<COPY>(l.src, l.len, l.dst, st, one);
        store_state(out + idx * 8, st);
    }
}

// graft_verify_split_kernel for a batch.
template <bool COPY, bool WIDE>
__global__ void __launch_bounds__(64) graft_batch_verify_split_kernel(const GraftBatchParams p,
                                                                      int64_t leaves_per_page,
                                                                      uint32_t *out, uint32_t one) {
    __shared__ SplitShared sm;
    const bool produce = split_begin(sm);
    if (p.write_meta) batch_metadata(p);
    const int lane = threadIdx.x & 31;
    const int64_t idx = split_chain<WIDE>(lane);
    const bool valid = idx < p.slice_jobs * p.n_layers * 2 * leaves_per_page;
    if (produce) {
        BatchLeaf l{nullptr, nullptr, 0};
        if (valid) l = batch_leaf<COPY>(p, idx, leaves_per_page);
        split_produce_leaf<COPY, WIDE>(sm, reinterpret_cast<const uint4 *>(l.src), reinterpret_cast<uint4 *>(l.dst),
                                       lane, one);
    } else {
        split_consume_leaf<WIDE>(sm, valid ? out + idx * 8 : nullptr, false, lane, one);
    }
}

// Whether the digest with state words st (written big-endian) differs from
// the 32 bytes at expected.
__device__ __forceinline__ bool digest_differs(const uint32_t st[8], const uint8_t *expected) {
    bool same = true;
#pragma unroll
    for (int k = 0; k < 32; ++k) same &= (uint8_t)(st[k >> 2] >> (24 - 8 * (k & 3))) == expected[k];
    return !same;
}

__device__ __forceinline__ void record_mismatch(DevStatus *status, int32_t page) {
    const int slot = atomicAdd(&status->n_mismatch, 1);
    if (slot < KVG_REPORT_MAX_PAGES) status->list[slot] = page;
    atomicCAS(&status->err, 0, (int32_t)KVG_ERR_DIGEST);
}

// What becomes of page p's digest.  PageOut: written to out and/or compared
// with expected; a mismatch is recorded in the status word.
struct PageOut {
    uint8_t *out;
    const uint8_t *expected;
    DevStatus *status;
    int32_t seq;
    __device__ __forceinline__ void operator()(int64_t p, const uint32_t st[8]) const {
        if (out) {
#pragma unroll
            for (int k = 0; k < 32; ++k) out[p * 32 + k] = (uint8_t)(st[k >> 2] >> (24 - 8 * (k & 3)));
        }
        if (expected && digest_differs(st, expected + p * 32)) {
            record_mismatch(status, (int32_t)p);
            status->seq = seq;
            status->batch_fail = 0;
        }
    }
};

// BatchCheck: page p of a batch's slice compared with its block's digest; the
// status keeps the last failing graft.
struct BatchCheck {
    const GraftJob *jobs;
    const GraftMeta *metas;
    int64_t job0, slice_jobs;
    uint32_t call;
    DevStatus *status;
    __device__ __forceinline__ void operator()(int64_t p, const uint32_t st[8]) const {
        const int64_t lkv = p / slice_jobs;
        const GraftJob job = jobs[job0 + p - lkv * slice_jobs];
        const GraftMeta &m = metas[job.meta];
        const int64_t page = lkv * job.block_pages + job.page;
        if (!digest_differs(st, m.digests + page * 32)) return;
        record_mismatch(status, (int32_t)page);
        atomicMax(&status->batch_fail, ((unsigned long long)call << 45) | ((unsigned long long)job.meta << 32) |
                                           (unsigned long long)(uint32_t)m.seq);
    }
};

// Page digest from its leaf digests: the message is the leaf digests' bytes,
// i.e. (big-endian) exactly the 8 state words of each leaf in order.
template <class Verdict>
__global__ void __launch_bounds__(128) sha256_pages_kernel(const uint32_t *leaf_words,
                                                           int64_t n_pages, int64_t m, const Verdict verdict,
                                                           uint32_t one) {
    after_previous();
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= n_pages) return;
    const uint32_t *lw = leaf_words + p * m * 8;
    uint32_t st[8];
    init_state(st);
    const int64_t nwords = m * 8;
    const int64_t nfull = nwords / 16;
    for (int64_t blk = 0; blk < nfull; ++blk) {
        uint32_t w[16];
        const uint4 *v = reinterpret_cast<const uint4 *>(lw + blk * 16);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
            const uint4 x = v[q];
            w[4 * q + 0] = x.x;
            w[4 * q + 1] = x.y;
            w[4 * q + 2] = x.z;
            w[4 * q + 3] = x.w;
        }
        compress<false>(st, w, one);
    }
    {
        uint32_t w[16];
#pragma unroll
        for (int q = 0; q < 16; ++q) w[q] = 0;
        const int remw = (int)(nwords - nfull * 16);  // 0 or 8
        for (int q = 0; q < remw; ++q) w[q] = lw[nfull * 16 + q];
        w[remw] = 0x80000000u;
        const uint64_t bits = (uint64_t)m * 32ull * 8ull;
        w[14] = (uint32_t)(bits >> 32);
        w[15] = (uint32_t)bits;
        compress<false>(st, w, one);
    }
    verdict(p, st);
}

// sha256_pages_kernel in the two-warp form: the loading warp feeds each page's
// leaf digests (already big-endian words) and the final block.
template <class Verdict>
__global__ void __launch_bounds__(64) sha256_pages_split_kernel(const uint32_t *leaf_words,
                                                                int64_t n_pages, int64_t m, const Verdict verdict,
                                                                uint32_t one) {
    __shared__ SplitShared sm;
    const bool produce = split_begin(sm);
    const int lane = threadIdx.x & 31;
    const int64_t p = (int64_t)blockIdx.x * kSplitChains + (lane & (kSplitChains - 1));
    const bool valid = p < n_pages;
    const int64_t nwords = m * 8;
    const int nfull = (int)(nwords / 16);
    const int remw = (int)(nwords - (int64_t)nfull * 16);  // 0 or 8
    if (produce) {
        const uint32_t *lw = leaf_words + (valid ? p : 0) * m * 8;
        const int half = lane / kSplitChains;
        // the lane's block of pair k: 16 whole words, the final block, or (past it) nothing
        uint4 nx[4];
        auto load = [&](int blk) {
#pragma unroll
            for (int q = 0; q < 4; ++q) nx[q] = make_uint4(0, 0, 0, 0);
            if (!valid) return;
            if (blk < nfull) {
#pragma unroll
                for (int q = 0; q < 4; ++q) nx[q] = reinterpret_cast<const uint4 *>(lw + (int64_t)blk * 16)[q];
            } else if (blk == nfull) {
                const uint64_t bits = (uint64_t)m * 32ull * 8ull;
                if (remw) {
                    nx[0] = reinterpret_cast<const uint4 *>(lw + (int64_t)nfull * 16)[0];
                    nx[1] = reinterpret_cast<const uint4 *>(lw + (int64_t)nfull * 16)[1];
                    nx[2].x = 0x80000000u;
                } else {
                    nx[0].x = 0x80000000u;
                }
                nx[3].z = (uint32_t)(bits >> 32);
                nx[3].w = (uint32_t)bits;
            }
        };
        const int n_pairs = (nfull + 2) >> 1;
        load(half);
        for (int k = 0; k < n_pairs; ++k) {
            uint32_t w[16];
#pragma unroll
            for (int q = 0; q < 4; ++q) {
                w[4 * q + 0] = nx[q].x;
                w[4 * q + 1] = nx[q].y;
                w[4 * q + 2] = nx[q].z;
                w[4 * q + 3] = nx[q].w;
            }
            if (k + 1 < n_pairs) load(2 * (k + 1) + half);
            split_hand_over(sm, w, k, lane, one);
        }
    } else {
        uint32_t st[4], full[8];
        split_consume(st, sm, nfull + 1, lane, one);
        split_whole_state(full, st);
        if (valid && lane < kSplitChains) verdict(p, full);
    }
}

// Streaming single-thread hasher for seg0 || seg1 of arbitrary lengths.
struct Stream {
    uint32_t one;
    uint32_t st[8];
    uint32_t w[16];
    int fill;  // bytes in w
    uint64_t total;

    __device__ void init(uint32_t one_) {
        one = one_;
        init_state(st);
        fill = 0;
        total = 0;
#pragma unroll
        for (int i = 0; i < 16; ++i) w[i] = 0;
    }
    __device__ void byte(uint8_t x) {
        w[fill >> 2] |= (uint32_t)x << (24 - 8 * (fill & 3));
        if (++fill == 64) {
            compress<false>(st, w, one);
            fill = 0;
#pragma unroll
            for (int i = 0; i < 16; ++i) w[i] = 0;
        }
    }
    __device__ void feed(const uint8_t *ptr, uint64_t n) {
        total += n;
        uint64_t k = 0;
        while (k < n && (fill != 0 || (reinterpret_cast<uintptr_t>(ptr + k) & 3))) byte(ptr[k++]);
        while (n - k >= 64) {
            const uint32_t *q = reinterpret_cast<const uint32_t *>(ptr + k);
#pragma unroll
            for (int i = 0; i < 16; ++i) w[i] = bswap(q[i]);
            compress<false>(st, w, one);
#pragma unroll
            for (int i = 0; i < 16; ++i) w[i] = 0;
            k += 64;
        }
        while (k < n) byte(ptr[k++]);
    }
    __device__ void final(uint8_t out[32]) {
        const uint64_t bits = total * 8ull;
        byte(0x80);
        while (fill != 56) byte(0);
        for (int i = 7; i >= 0; --i) byte((uint8_t)(bits >> (8 * i)));
        for (int k = 0; k < 8; ++k) {
            out[4 * k + 0] = (uint8_t)(st[k] >> 24);
            out[4 * k + 1] = (uint8_t)(st[k] >> 16);
            out[4 * k + 2] = (uint8_t)(st[k] >> 8);
            out[4 * k + 3] = (uint8_t)st[k];
        }
    }
};

// SHA-256 of seg0 || seg1: one serial chain, run by lane 0 of one warp.
// When both segments are 4-byte aligned and seg0's length is a multiple of 4
// (a block's position tags and page digests are), the 32 lanes load the next
// 2 KiB of the message (coalesced 4-byte words) while lane 0 compresses the
// current 2 KiB from shared memory, so the chain never waits on a load;
// otherwise (any byte alignment) lane 0 streams the bytes itself.
constexpr int kSerialChunkWords = 512;  // 2 KiB = 32 blocks per chunk

__device__ __forceinline__ uint32_t msg_word(const uint8_t *seg0, uint64_t n0, const uint8_t *seg1, uint64_t i) {
    const uint64_t off = 4 * i;
    return off < n0 ? *reinterpret_cast<const uint32_t *>(seg0 + off)
                    : *reinterpret_cast<const uint32_t *>(seg1 + (off - n0));
}

__global__ void __launch_bounds__(32) sha256_serial_kernel(const uint8_t *seg0, uint64_t n0, const uint8_t *seg1,
                                                           uint64_t n1, uint8_t *out, const uint8_t *expected,
                                                           DevStatus *status, uint32_t one) {
    after_previous();
    __shared__ uint32_t buf[2][kSerialChunkWords];
    const int lane = threadIdx.x;
    if (blockIdx.x != 0) return;
    const uint64_t total = n0 + n1;
    const bool fast = !((reinterpret_cast<uintptr_t>(seg0) | reinterpret_cast<uintptr_t>(seg1) | n0) & 3);
    const uint64_t n_chunks = fast ? total / (4 * kSerialChunkWords) : 0;
    Stream s;
    if (lane == 0) s.init(one);
    if (n_chunks) {
        for (int k = 0; k < kSerialChunkWords / 32; ++k)
            buf[0][lane + 32 * k] = msg_word(seg0, n0, seg1, lane + 32 * k);
        __syncwarp();
        for (uint64_t c = 0; c < n_chunks; ++c) {
            uint32_t nxt[kSerialChunkWords / 32];
            const bool more = c + 1 < n_chunks;
            if (more) {
#pragma unroll
                for (int k = 0; k < kSerialChunkWords / 32; ++k)
                    nxt[k] = msg_word(seg0, n0, seg1, (c + 1) * kSerialChunkWords + lane + 32 * k);
            }
            if (lane == 0) {
                const uint32_t *cur = buf[c & 1];
                for (int b = 0; b < kSerialChunkWords / 16; ++b) {
                    uint32_t w[16];
#pragma unroll
                    for (int i = 0; i < 16; ++i) w[i] = bswap(cur[16 * b + i]);
                    compress<false>(s.st, w, one);
                }
            }
            __syncwarp();
            if (more) {
#pragma unroll
                for (int k = 0; k < kSerialChunkWords / 32; ++k) buf[(c + 1) & 1][lane + 32 * k] = nxt[k];
            }
            __syncwarp();
        }
    }
    if (lane != 0) return;
    // the rest of the message (and all of it on the byte path)
    const uint64_t done = n_chunks * 4 * kSerialChunkWords;
    s.total = done;
    if (done < n0) s.feed(seg0 + done, n0 - done);
    const uint64_t d1 = done > n0 ? done - n0 : 0;
    if (d1 < n1) s.feed(seg1 + d1, n1 - d1);
    uint8_t dg[32];
    s.final(dg);
    if (out)
        for (int k = 0; k < 32; ++k) out[k] = dg[k];
    if (expected) {
        bool same = true;
        for (int k = 0; k < 32; ++k) same &= dg[k] == expected[k];
        if (!same) {
            atomicAdd(&status->n_mismatch, 1);
            atomicCAS(&status->err, 0, (int32_t)KVG_ERR_DIGEST);
        }
    }
}

// sha256_serial_kernel in the two-warp form: every pair of lanes of the
// rounds' warp runs the same chain (lane 0's result is kept) and the other warp reads the message
// two pairs of blocks ahead, the padding included.  For 4-byte aligned
// segments with seg0's length a multiple of 4.
// Word i of the padded message of n_blocks blocks, big-endian.
__device__ __forceinline__ uint32_t padded_word(const uint8_t *seg0, uint64_t n0, const uint8_t *seg1, uint64_t n1,
                                                uint64_t n_blocks, uint64_t i) {
    const uint64_t total = n0 + n1, off = 4 * i;
    if (off + 4 <= total) return bswap(msg_word(seg0, n0, seg1, i));
    if (i + 2 >= 16 * n_blocks) {
        const uint64_t bits = total * 8ull;
        return i + 2 == 16 * n_blocks ? (uint32_t)(bits >> 32) : i + 1 == 16 * n_blocks ? (uint32_t)bits : 0u;
    }
    uint32_t v = 0;
    for (int b = 0; b < 4; ++b) {
        const uint64_t at = off + b;
        const uint32_t x = at < total ? (at < n0 ? seg0[at] : seg1[at - n0]) : at == total ? 0x80u : 0u;
        v |= x << (24 - 8 * b);
    }
    return v;
}

// Blocks [b0, b1) of the padded message's n_blocks, from the state `from`
// (b0 > 0).  The part that ends the message writes the digest to out and/or
// compares it with expected; the others write the state to `to`.
__global__ void __launch_bounds__(64) sha256_serial_split_kernel(const uint8_t *seg0, uint64_t n0, const uint8_t *seg1,
                                                                 uint64_t n1, int32_t b0, int32_t b1,
                                                                 int32_t n_blocks, const uint32_t *from, uint32_t *to,
                                                                 uint8_t *out, const uint8_t *expected,
                                                                 DevStatus *status, uint32_t one) {
    __shared__ SplitShared sm;
    const bool produce = split_begin(sm);
    const int lane = threadIdx.x & 31;
    if (blockIdx.x != 0) return;
    if (produce) {
        const uint64_t whole = (n0 + n1) / 64;  // blocks without padding
        uint32_t n1w[16], n2w[16];
        // block blk as big-endian words (past the part: zeros)
        auto load = [&](uint32_t w[16], int blk) {
            if (blk >= b1) {
#pragma unroll
                for (int i = 0; i < 16; ++i) w[i] = 0u;
            } else if ((uint64_t)blk < whole) {
#pragma unroll
                for (int i = 0; i < 16; ++i) w[i] = bswap(msg_word(seg0, n0, seg1, 16ull * blk + i));
            } else {
#pragma unroll
                for (int i = 0; i < 16; ++i) w[i] = padded_word(seg0, n0, seg1, n1, n_blocks, 16ull * blk + i);
            }
        };
        const int first = b0 + lane / kSplitChains;
        const int n_pairs = (b1 - b0 + 1) >> 1;
        load(n1w, first);
        load(n2w, first + 2);
        for (int k = 0; k < n_pairs; ++k) {
            uint32_t w[16];
#pragma unroll
            for (int i = 0; i < 16; ++i) {
                w[i] = n1w[i];
                n1w[i] = n2w[i];
            }
            if (k + 2 < n_pairs) load(n2w, first + 2 * (k + 2));
            split_hand_over(sm, w, k, lane, one);
        }
        return;
    }
    uint32_t st[4], full[8];
    split_consume(st, sm, b1 - b0, lane, one, b0 > 0 ? from : nullptr);
    split_whole_state(full, st);
    if (lane != 0) return;
    if (b1 < n_blocks) {
        store_state(to, full);
        return;
    }
    if (out) {
#pragma unroll
        for (int k = 0; k < 8; ++k) reinterpret_cast<uint32_t *>(out)[k] = bswap(full[k]);
    }
    if (expected && digest_differs(full, expected)) {
        atomicAdd(&status->n_mismatch, 1);
        atomicCAS(&status->err, 0, (int32_t)KVG_ERR_DIGEST);
    }
}

}  // namespace

// The two-warp form is used for pages of whole 4 KiB leaves (leaf launches
// below) and for page digests, which read their input from L2, up to eight of
// its CTAs per SM; beyond that the one-warp forms keep more chains going per
// SM.  KVG_SHA_NO_SPLIT=1 turns it off.
static bool split_off() {
    static const bool off = env_knob("KVG_SHA_NO_SPLIT", 0) > 0;
    return off;
}

// Leaves per SM up to which a leaf launch takes the two-warp form.  Up to two
// CTAs of 16 chains per SM (four warps, one per scheduler) a chain has two
// lanes; from there to two CTAs of 32 the wide form is faster: digests of 16,
// 32, 48 and 64 leaves per SM take 71, 73, 87 and 92 us with two lanes, 73, 75,
// 74 and 76 wide, and 104 to 109 in one warp; of 96 and 128, 138 and 176, 124
// and 127, and 110.  A verified graft from pinned host memory keeps the one-warp
// form: its leaf loads outlast the rounds of a block here (the last chunk of
// the 12B block's host-store graft, 40 leaves per SM, made the e2e step
// 15.73-15.83 ms instead of 15.63-15.71).
static int split_leaves_per_sm() {
    static const int v = env_knob("KVG_SHA_SPLIT_LEAVES_PER_SM", 2 * kWideChains);
    return v;
}
static bool split_wide(int64_t n, int n_sm) { return n > (int64_t)n_sm * 2 * kSplitChains; }
static int split_grid(int64_t n, bool wide) {
    const int per = wide ? kWideChains : kSplitChains;
    return (int)((n + per - 1) / per);
}

// Whether a one-warp launch of sha256_leaves_kernel uses the latency order of
// additions: checking a restored block of 107, 215, 323, 431 and 646 leaves per
// SM takes 127, 201, 278, 350 and 499 us with it, 138, 217, 290, 364 and 507
// without; of 1,024 and more the same either way.  (In the copying kernels it
// costs more registers than it gains: 198 against 146 us at 107 leaves per SM.)
static bool lat_order(int64_t n, int n_sm) {
    static const int per_sm = env_knob("KVG_SHA_LAT_LEAVES_PER_SM", 512);
    return n <= (int64_t)n_sm * per_sm;
}

// Whether a leaf launch may start while the kernel before it still holds SMs.
// Not where it has a CTA for more than every fourth SM and at most four for
// each: its CTAs are then placed around the other's (the page digests of the
// call before), some SMs get one more than their share, and the chains there are
// what the launch waits for.  Digests of 64 KiB pages back to back, us a call, 48,
// 64, 128, 220 and 512 leaves per SM: 65, 109, 156, 240 and 386 started early, 68,
// 68, 98, 173 and 325 not; of 4 KiB pages with 48 leaves per SM 103 and 62.  A few
// CTAs gain the 3 us of the launch (20 leaves per SM: 63 against 66).
static bool leaves_early(int64_t grid, int n_sm) { return grid * 4 <= n_sm || grid > (int64_t)n_sm * 4; }

static int current_sm_count() {
    static int cache[64] = {};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return 0;
    if (!cache[dev]) cudaDeviceGetAttribute(&cache[dev], cudaDevAttrMultiProcessorCount, dev);
    return cache[dev];
}

static bool regs_only() {
    static const bool v = env_knob("KVG_SHA_REGISTER_FORM", 0) > 0;
    return v;
}

cudaError_t launch_sha256_leaves(const PageSource &src, int64_t n_pages, uint32_t *leaf_words,
                                 int n_sm, cudaStream_t s, bool split_ok, int max_ctas) {
    const int64_t m = (int64_t)((src.page_bytes + kLeafBytes - 1) / kLeafBytes);
    const int64_t n = n_pages * m;
    if (n == 0) return cudaSuccess;
    if (split_ok && !split_off() && src.page_bytes % kLeafBytes == 0 && n <= (int64_t)n_sm * split_leaves_per_sm()) {
        const bool wide = split_wide(n, n_sm);
        auto *kernel = wide ? sha256_leaves_split_kernel<true> : sha256_leaves_split_kernel<false>;
        const int grid = split_grid(n, wide);
        return launch_kernel(leaves_early(grid, n_sm), kernel, grid, 64, 0, s, src, n_pages, m, leaf_words, 1u);
    }
    int64_t grid = (n + 127) / 128;
    // One CTA per 128 leaves (no grid-stride cap by default): 4 CTAs of
    // 125 registers are resident per SM and the rest queue, which measured
    // 2-3% faster than a capped, striding grid.
    static const int ctas_per_sm = env_knob("KVG_SHA_CTAS_PER_SM", 0);
    if (ctas_per_sm > 0 && grid > (int64_t)n_sm * ctas_per_sm) grid = (int64_t)n_sm * ctas_per_sm;
    if (max_ctas > 0 && grid > max_ctas) grid = max_ctas;
    auto *kernel = lat_order(n, n_sm) ? sha256_leaves_kernel<true> : sha256_leaves_kernel<false>;
    return launch_kernel(leaves_early(grid, n_sm), kernel, (int)grid, 128, 0, s, src, n_pages, m, leaf_words, 1u);
}

cudaError_t launch_graft_verify(const GraftParams &p, uint32_t *leaf_words, int n_sm, cudaStream_t s, bool ring_ok,
                                bool split_ok) {
    const int64_t m = (int64_t)((p.page_bytes + kLeafBytes - 1) / kLeafBytes);
    const int64_t n = (int64_t)p.n_layers * 2 * p.npb * m;
    if (n == 0) return cudaSuccess;
    if (split_ok && !split_off() && p.page_bytes % kLeafBytes == 0 && n <= (int64_t)n_sm * split_leaves_per_sm()) {
        const bool wide = split_wide(n, n_sm);
        auto *kernel = wide ? graft_verify_split_kernel<true> : graft_verify_split_kernel<false>;
        const int grid = split_grid(n, wide);
        return launch_kernel(leaves_early(grid, n_sm), kernel, grid, 64, 0, s, p, m, leaf_words, 1u);
    }
    int64_t grid = (n + 127) / 128;
    // One CTA per 128 leaves (no grid-stride cap by default): four CTAs of
    // the register form (125 registers) or five of the ring form (96) are
    // resident per SM and the rest queue.
    static const int ctas_per_sm = env_knob("KVG_SHA_CTAS_PER_SM", 0);
    if (ctas_per_sm > 0 && grid > (int64_t)n_sm * ctas_per_sm) grid = (int64_t)n_sm * ctas_per_sm;
    // a full wave of the ring form (five CTAs on every SM) or more, where the
    // caller allows it: the ring form; otherwise the register form (see
    // graft_verify_ring_kernel).  KVG_SHA_REGISTER_FORM=1 keeps the register
    // form for every size.
    if (ring_ok && !regs_only() && n >= (int64_t)n_sm * 5 * 128 && grid > (int64_t)n_sm * 4) {
        const size_t smem = (size_t)128 * kGraftVerifyRing * 64;  // 24 KiB of ring slots per CTA
        return launch_after(graft_verify_ring_kernel, (int)grid, 128, smem, s, p, m, leaf_words, 1u);
    }
    return launch_kernel(leaves_early(grid, n_sm), graft_verify_kernel, (int)grid, 128, 0, s, p, m, leaf_words, 1u);
}

cudaError_t launch_graft_batch_verify(const GraftBatchParams &p, uint32_t *leaf_words, int n_sm, cudaStream_t s,
                                      bool ring_ok) {
    const int64_t m = (int64_t)((p.page_bytes + kLeafBytes - 1) / kLeafBytes);
    const int64_t n = p.slice_jobs * p.n_layers * 2 * m;
    if (n == 0) return cudaSuccess;
    const int grid = (int)((n + 127) / 128);
    // The forms and their launch sizes are those of launch_graft_verify, the two-warp
    // form also where re-based pages are hashed in pinned host memory: one graft of
    // 40 tokens of 2 layers of the tiny shape 94 us (one warp 187), 4 of 200 tokens of
    // the 12B shape, 27 leaves per SM, 244 (293).
    if (!split_off() && p.page_bytes % kLeafBytes == 0 && n <= (int64_t)n_sm * split_leaves_per_sm()) {
        const bool wide = split_wide(n, n_sm);
        auto *kernel = p.hash_only ? (wide ? graft_batch_verify_split_kernel<false, true>
                                           : graft_batch_verify_split_kernel<false, false>)
                                   : (wide ? graft_batch_verify_split_kernel<true, true>
                                           : graft_batch_verify_split_kernel<true, false>);
        return launch_after(kernel, split_grid(n, wide), 64, 0, s, p, m, leaf_words, 1u);
    }
    if (ring_ok && !p.hash_only && !regs_only() && n >= (int64_t)n_sm * 5 * 128) {
        const size_t smem = (size_t)128 * kGraftVerifyRing * 64;
        return launch_after(graft_batch_verify_ring_kernel, grid, 128, smem, s, p, m, leaf_words, 1u);
    }
    return launch_after(p.hash_only ? graft_batch_verify_kernel<false> : graft_batch_verify_kernel<true>, grid, 128, 0,
                        s, p, m, leaf_words, 1u);
}

template <class Verdict>
static cudaError_t launch_pages(const uint32_t *leaf_words, int64_t n_pages, int64_t leaves_per_page,
                                const Verdict &verdict, cudaStream_t s) {
    if (n_pages == 0) return cudaSuccess;
    if (!split_off() && n_pages <= (int64_t)current_sm_count() * 8 * kSplitChains)
        return launch_after(sha256_pages_split_kernel<Verdict>, (int)((n_pages + kSplitChains - 1) / kSplitChains), 64,
                            0, s, leaf_words, n_pages, leaves_per_page, verdict, 1u);
    return launch_after(sha256_pages_kernel<Verdict>, (int)((n_pages + 127) / 128), 128, 0, s, leaf_words, n_pages,
                        leaves_per_page, verdict, 1u);
}

cudaError_t launch_sha256_pages(const uint32_t *leaf_words, int64_t n_pages, int64_t leaves_per_page,
                                uint8_t *out, const uint8_t *expected, DevStatus *status,
                                int32_t seq, cudaStream_t s) {
    return launch_pages(leaf_words, n_pages, leaves_per_page, PageOut{out, expected, status, seq}, s);
}

cudaError_t launch_graft_batch_pages(const GraftBatchParams &p, const uint32_t *leaf_words, DevStatus *status,
                                     uint32_t call, cudaStream_t s) {
    const int64_t m = (int64_t)((p.page_bytes + kLeafBytes - 1) / kLeafBytes);
    return launch_pages(leaf_words, p.slice_jobs * p.n_layers * 2, m,
                        BatchCheck{p.jobs, p.metas, p.job0, p.slice_jobs, call, status}, s);
}

int64_t serial_blocks(uint64_t bytes) { return (int64_t)((bytes + 9 + 63) / 64); }
bool sha256_parts_ok() { return !split_off(); }

cudaError_t launch_sha256_serial(const uint8_t *seg0, uint64_t n0, const uint8_t *seg1, uint64_t n1,
                                 uint8_t *out, const uint8_t *expected, DevStatus *status,
                                 cudaStream_t s) {
    const bool aligned = !((reinterpret_cast<uintptr_t>(seg0) | reinterpret_cast<uintptr_t>(seg1) |
                            reinterpret_cast<uintptr_t>(out) | n0) & 3);
    const int64_t n_blocks = serial_blocks(n0 + n1);
    if (!split_off() && aligned && n_blocks < (1ll << 30)) {
        sha256_serial_split_kernel<<<1, 64, 0, s>>>(seg0, n0, seg1, n1, 0, (int32_t)n_blocks, (int32_t)n_blocks,
                                                    nullptr, nullptr, out, expected, status, 1u);
    } else {
        sha256_serial_kernel<<<1, 32, 0, s>>>(seg0, n0, seg1, n1, out, expected, status, 1u);
    }
    count_launches(1);
    return cudaGetLastError();
}

cudaError_t launch_sha256_serial_part(const uint8_t *seg0, uint64_t n0, const uint8_t *seg1, uint64_t n1, int64_t b0,
                                      int64_t b1, uint8_t *state, uint8_t *out, cudaStream_t s) {
    if (b1 <= b0) return cudaSuccess;
    sha256_serial_split_kernel<<<1, 64, 0, s>>>(seg0, n0, seg1, n1, (int32_t)b0, (int32_t)b1,
                                                (int32_t)serial_blocks(n0 + n1),
                                                reinterpret_cast<const uint32_t *>(state),
                                                reinterpret_cast<uint32_t *>(state), out, nullptr, nullptr, 1u);
    count_launches(1);
    return cudaGetLastError();
}

}  // namespace kvg
