// init_tc.cu -- exhaustive nearest-neighbour initialisation at the coarsest
// level (Sec. III-D; every seed starts from the target centre of least patch
// distance, Eq. 3, ties to the smaller raster index) on the tensor cores, for
// the squared-L2 cost.
//
// Over integers D(s, q) = sum |a|^2 + sum |b|^2 - 2 X(s, q), and the cross
// terms of all seeds against all target centres form one dense contraction
//   X(s, q) = sum_k A(s, k) B(q, k),   k = (patch row r, column p, channel).
// tcgen05.mma (kind::f16) multiplies fp16 operands from shared memory into
// fp32 accumulators in tensor memory.  To make that exact, every descriptor
// value v (|v| <= 12240, Sobel-5 on 8-bit channels) is split as
// v = 128 v_h + v_l with v_l in [-64, 63] and v_h in [-96, 96], both exact in
// fp16, and
//   X = 2^14 <a_h, b_h> + 2^7 (<a_h, b_l> + <a_l, b_h>) + <a_l, b_l>
// takes three accumulators.  Each product is an integer of magnitude at most
// 96 * 96 (one accumulator) or 2 * 96 * 64 (the middle one, two products per
// element), so for patches up to 15 x 15 x 6 every partial sum is an integer
// below 2^24 (225 * 6 * 12288 = 16588800) and fp32 holds it exactly.
//
// No operand is copied out patch by patch.  A staged unit is 16 bytes, eight
// fp16 values: a colour pixel (six channels and two zero pads), or a run of
// four gray pixels from a column on (two channels each; the runs of
// neighbouring columns overlap).  One MMA step (K = 16) is two units, and the
// tensor core reads an operand as groups of eight 16-byte rows, 16 bytes
// apart, the groups 128 bytes apart, the second 8-value half of the step at a
// free distance (the descriptor's leading-byte offset):
// - target centres, flattened as n = y Wt + x over a copy of the target with a
//   border of P / 2 on every side (row pitch Wt = tw + P - 1): unit (p, r) of
//   centre n is staged unit n + r Wt + p, so consecutive centres are
//   consecutive rows of every step;
// - seeds, on a lattice of stride sigma: the reference is staged as sigma^2
//   phase images R_{phi,psi}(u, v) = R(sigma u + phi + o, sigma v + psi + o),
//   o = c - P / 2, of row pitch Wu = nx + (P - 1) / sigma; seed (i, j),
//   flattened as m = j Wu + i, reads unit (p, r) in phase
//   (p mod sigma, r mod sigma) at m + (r div sigma) Wu + p div sigma, so
//   consecutive seeds are again consecutive rows.
// The two units of a step are any two whose staged addresses increase in both
// operands; a unit left without a partner takes a block of zeros on the target
// side.  Flattened seeds with i >= nx and centres with x >= tw are computed
// and ignored.  A gray patch row is ceil(P / 4) runs; where P is no multiple
// of four the last run's pixels past the patch must not count, so the seeds
// read it from a second copy of the phase images in which they are zero.
//
// A tile is 128 flattened seeds (the MMA's M, one tensor-memory lane each)
// against 160 flattened centres (the MMA's N; three fp32 accumulators of 160
// columns).  Only the rows that a tile reads are staged: patch row r of the
// tile's centres is one run of 160 + P - 1 units, and phase row q of its seeds
// one of 128 + e + 1 (e = (P - 1) / sigma); where the image is narrower than
// such a run, the runs overlap and are staged once, at the image's own pitch.
// Where all rows of the patch fit in shared memory (TC_SMEM) they are staged
// once for TC_NT neighbouring tiles; a patch over a wider or denser lattice
// is cut into chunks of sigma rows, staged in turn into two buffers, the
// accumulators running over the chunks.
//
// A CTA takes one seed tile and a band of centre tiles of one direction of
// one pair.  Eight worker warps stage and convert; one more warp issues the
// MMAs of a staged chunk (one thread) and commits them to the buffer's
// mbarrier, so that the next chunk is staged while they run; after a tile's
// last chunk every worker warp reads its lanes' accumulators (warp w: lanes
// 32 (w mod 4) .., columns 80 (w div 4) ..), forms the exact costs and keeps
// per seed the least (cost, raster index), packed as cost << 24 | q (cost <
// 2^40 for these patches, q < 2^24).  The bands of a seed meet in an atomicMin
// on its cost word, cleared before and unpacked after.
#include <cuda_fp16.h>

#include <algorithm>
#include <cstring>

#include "match_common.cuh"

namespace pgm {

long long wait_limit();      // the mbarrier wait limit (pgm_set_wait_limit)

namespace {

constexpr int TC_M = 128;              // flattened seeds per tile
constexpr int TC_N = 160;              // flattened target centres per tile
constexpr int TC_NT = 2;               // centre tiles per CTA, whole patches staged, and
constexpr int TC_NTC = 4;              // patches staged in chunks; one each for a small grid
constexpr int TC_WORKERS = 8;          // staging and epilogue warps
constexpr int TC_THREADS = 32 * (TC_WORKERS + 1);
constexpr int TC_MAXP = 15;            // the exact-accumulation bound above
constexpr int TC_MAXSTEP = 128;        // K steps of a 15 x 15 patch: 113, in chunks at most 120
constexpr int TC_HDR = 8;              // header units: mbarriers, tensor-memory address, abort
constexpr int TC_TMEM_COLS = 512;      // 3 x 160 accumulator columns, rounded to a power of 2
constexpr int TC_SMEM = 200 * 1024;    // shared memory of one CTA at most
constexpr long long TC_DRAIN_CYCLES = 1ll << 31;

// The K steps of each direction's patch, chunk after chunk (first step of
// chunk c: n0[c]); a chunk is Q sigma patch rows.
struct TcSteps {
    int nchunk[2], Q[2], per[2];       // per: centre tiles per CTA
    int n0[2][TC_MAXP + 1];
    uint16_t pr[2][TC_MAXSTEP];        // p1 | r1 << 4 | p2 << 8 | r2 << 12; p2 = 15: zero partner
};

struct TcGeom {
    int e, Wu, mtiles, pa, LA, copies; // seeds: row pitch, tiles, staged pitch, units per phase slice
    int Wt, ntiles, pb, LB;            // centres
    int NT, bands, ctas, phases, bufs, buf_units;
};

// Q: phase rows per chunk, nchunk chunks; gray: the runs' second copy
__host__ __device__ inline TcGeom tc_geom(const DirLvl& D, int sigma, int Q, int nchunk, int per,
                                          bool gray) {
    TcGeom g;
    const int P = D.P;
    g.e = (P - 1) / sigma;
    g.phases = sigma * sigma;
    g.Wu = D.nx + g.e;
    g.mtiles = (D.ny * g.Wu + TC_M - 1) / TC_M;
    const int ra = TC_M + g.e + 1;                     // one run; + 1: a zero partner's rows
    g.pa = g.Wu < ra ? g.Wu : ra;
    g.LA = g.pa * (Q - 1) + ra;
    g.copies = gray && P % 4 ? 2 : 1;
    g.NT = nchunk > 1 ? 1 : per;                       // tiles staged together
    g.Wt = D.tw + P - 1;
    g.ntiles = (D.th * g.Wt + TC_N - 1) / TC_N;
    const int rb = g.NT * TC_N + P - 1, rows = Q * sigma < P ? Q * sigma : P;
    g.pb = g.Wt < rb ? g.Wt : rb;
    g.LB = g.pb * (rows - 1) + rb;
    g.bands = (g.ntiles + per - 1) / per;
    g.ctas = g.mtiles * g.bands;
    g.bufs = nchunk > 1 ? 2 : 1;
    g.buf_units = 2 * g.copies * g.phases * g.LA + 2 * g.LB;
    return g;
}

// shared memory in 16-byte units: header, centre table (sum |b|^2 and raster
// index per column), K-step table, staging buffers (reference phase slices,
// high then low parts; target rows, high then low), zero block, per-seed
// results of the two column halves
__host__ __device__ inline int tc_units(const TcGeom& g) {
    return TC_HDR + TC_NT * TC_N + TC_MAXSTEP + g.bufs * g.buf_units + TC_N + 2 * TC_M / 2;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
    return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void tc_mbar_init(uint32_t bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ bool tc_mbar_test(uint32_t bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok) : "r"(bar), "r"(parity) : "memory");
    return ok != 0;
}
// wait for phase `parity`; false after `limit` cycles or once another warp has
// flagged an abort
__device__ __forceinline__ bool tc_mbar_wait(uint32_t bar, uint32_t parity, long long limit,
                                             const volatile int* abort) {
    const long long t0 = clock64();
    for (;;) {
        if (tc_mbar_test(bar, parity)) return true;
        if (abort && *abort) return false;
        if (clock64() - t0 > limit) return false;
    }
}
__device__ __forceinline__ void tc_mbar_arrive(uint32_t bar) {
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tc_fence_before() {
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
}
// K-major operand without swizzling: groups of eight 16-byte rows, 128 bytes
// apart (stride-dimension offset); the second 8-value half of the step `lbo`
// bytes after the first (leading-dimension offset); descriptor version 1
__device__ __forceinline__ uint64_t tc_desc(uint32_t addr, uint32_t lbo) {
    return (uint64_t)((addr >> 4) & 0x3fffu) | ((uint64_t)((lbo >> 4) & 0x3fffu) << 16) |
           ((uint64_t)(128u >> 4) << 32) | (1ull << 46);
}
// D[tmem] (+)= A B^T for one K step of 16; accumulate = 0 overwrites
__device__ __forceinline__ void tc_mma(uint32_t tmem, uint64_t a, uint64_t b, uint32_t idesc,
                                       uint32_t accumulate) {
    asm volatile(
        "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
        " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n"
        ::"r"(tmem), "l"(a), "l"(b), "r"(idesc), "r"(accumulate) : "memory");
}
// arrive on the mbarrier once every MMA this thread issued has completed
__device__ __forceinline__ void tc_commit(uint32_t bar) {
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n"
                 ::"r"(bar) : "memory");
}
// 16 consecutive accumulator columns of this thread's lane (32-bit each),
// waited for before the registers are used
__device__ __forceinline__ void tc_ld16(uint32_t taddr, uint32_t (&v)[16]) {
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
        "%11, %12, %13, %14, %15}, [%16];\n"
        "tcgen05.wait::ld.sync.aligned;\n"
        : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
          "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]),
          "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
        : "r"(taddr) : "memory");
}

// the eight int16 of a unit as fp16 high and low parts, v = 128 v_h + v_l.
// Both parts plus 128 lie in [32, 255], so 1024 + 128 + part is the fp16 with
// bits 0x6400 | (part + 128), and one packed subtraction of 1152 leaves the
// part (exact); cheaper than two conversions per value.
__device__ __forceinline__ void tc_split(const uint4 w, uint4& hi, uint4& lo) {
    const uint32_t in[4] = {w.x, w.y, w.z, w.w};
    uint32_t h[4], l[4];
    const __half2 off = __halves2half2(__ushort_as_half(0x6480), __ushort_as_half(0x6480));   // 1152
#pragma unroll
    for (int i = 0; i < 4; ++i) {
        // per 16-bit half: t = v + 64 + 16384 (in [4208, 28688]); the low 7
        // bits are v_l + 64, the others v_h + 128
        const uint32_t t = __vadd2(in[i], 0x40404040u);
        const uint32_t lb = (t & 0x007f007fu) + 0x64406440u;          // 0x6400 | (v_l + 128)
        const uint32_t hb = ((t >> 7) & 0x01ff01ffu) + 0x64006400u;   // 0x6400 | (v_h + 128)
        const __half2 lv = __hsub2(*reinterpret_cast<const __half2*>(&lb), off);
        const __half2 hv = __hsub2(*reinterpret_cast<const __half2*>(&hb), off);
        l[i] = *reinterpret_cast<const uint32_t*>(&lv);
        h[i] = *reinterpret_cast<const uint32_t*>(&hv);
    }
    hi = make_uint4(h[0], h[1], h[2], h[3]);
    lo = make_uint4(l[0], l[1], l[2], l[3]);
}

// the unit at pixel (X, Y), clamped to the padded image: the colour pixel
// there, or the gray pixels X .. X + 3 (each clamped); keep < 4: only the
// first `keep` of them
template <bool GRAY>
__device__ __forceinline__ uint4 tc_unit(const int16_t* img, int pitch, int w, int h, int X, int Y,
                                         int keep) {
    const int y = clampi(Y, -BORD, h + BORD - 1);
    const int16_t* row = img + (ptrdiff_t)y * pitch;
    if constexpr (!GRAY) {
        (void)keep;
        const int x = clampi(X, -BORD, w + BORD - 1);
        return __ldg(reinterpret_cast<const uint4*>(row + 8 * (ptrdiff_t)x));
    } else {
        uint32_t v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const int x = clampi(X + k, -BORD, w + BORD - 1);
            v[k] = k < keep ? __ldg(reinterpret_cast<const uint32_t*>(row) + x) : 0u;
        }
        return make_uint4(v[0], v[1], v[2], v[3]);
    }
}

template <bool GRAY>
__global__ void __launch_bounds__(TC_THREADS, 1)
k_init_tc(const __grid_constant__ LvlBatch B, const MatchConst mc, const __grid_constant__ TcSteps T,
          long long limit) {
    extern __shared__ __align__(1024) uint4 sm4[];
    const int dir = blockIdx.z, pair = blockIdx.y;
    const DirLvl& D = B.d[pair][dir];
    const int sg = mc.sigma, P = D.P, h = P / 2;
    const int nchunk = T.nchunk[dir], Q = T.Q[dir];
    const int per = T.per[dir];
    const TcGeom g = tc_geom(D, sg, Q, nchunk, per, GRAY);
    if ((int)blockIdx.x >= g.ctas || D.nx * D.ny == 0) return;
    const int mt = blockIdx.x % g.mtiles, band = blockIdx.x / g.mtiles;
    const int m0 = mt * TC_M;
    const int tile0 = band * per, ntile = min(per, g.ntiles - tile0);
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int tail = 4 * ((P - 1) / 4);                // first column of a gray row's last run

    // shared memory, in 16-byte units
    uint4* sQ = sm4 + TC_HDR;                          // centre table of one tile (two: halves)
    uint4* sS = sQ + TC_NT * TC_N;                     // K steps: a1, a2 - a1, b1, b2 - b1 (-1: zero)
    uint4* sBuf = sS + TC_MAXSTEP;
    uint4* sZ = sBuf + g.bufs * g.buf_units;           // TC_N zero rows
    unsigned long long* sBest = reinterpret_cast<unsigned long long*>(sZ + TC_N);   // [2][TC_M]
    const uint32_t bar_full = smem_u32(sm4), bar_done = bar_full + 16, bar_acc = bar_full + 32,
                   bar_tab = bar_full + 48;
    uint32_t* s_tmem = reinterpret_cast<uint32_t*>(sm4) + 10;
    volatile int* s_abort = reinterpret_cast<volatile int*>(sm4) + 11;
    const int hl_a = g.copies * g.phases * g.LA;       // units from the high to the low parts
    const int off_b = 2 * hl_a;

    if (tid == 0) {
        for (int b = 0; b < 2; ++b) {
            tc_mbar_init(bar_full + 8 * b, TC_WORKERS);
            tc_mbar_init(bar_done + 8 * b, 1);
        }
        tc_mbar_init(bar_acc, TC_WORKERS);
        tc_mbar_init(bar_tab, TC_WORKERS);
        *s_abort = 0;
        asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    if (warp == TC_WORKERS) {                          // the accumulators: 512 columns, all lanes
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n"
                     ::"r"(smem_u32(s_tmem)), "r"(TC_TMEM_COLS) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
    }
    for (int k = tid; k < TC_N; k += TC_THREADS) sZ[k] = make_uint4(0u, 0u, 0u, 0u);
    // K steps: offsets (units) of both halves in both operands of a buffer
    for (int t = tid; t < T.n0[dir][nchunk]; t += TC_THREADS) {
        int c = 0;
        while (T.n0[dir][c + 1] <= t) ++c;
        const int ra = c * Q * sg;                     // the chunk's first patch row
        const uint32_t s = T.pr[dir][t];
        auto aoff = [&](int p, int r) {
            const int copy = GRAY && g.copies == 2 && p == tail;
            return ((copy * sg + r % sg) * sg + p % sg) * g.LA + ((r - ra) / sg) * g.pa + p / sg;
        };
        const int p1 = s & 15, r1 = (s >> 4) & 15, p2 = (s >> 8) & 15, r2 = s >> 12;
        const bool z = p2 == 15;
        const int a1 = aoff(p1, r1), b1 = (r1 - ra) * g.pb + p1;
        const int a2 = z ? a1 + 1 : aoff(p2, r2);
        sS[t] = make_uint4((uint32_t)a1, (uint32_t)(a2 - a1), (uint32_t)b1,
                           z ? 0xffffffffu : (uint32_t)((r2 - ra) * g.pb + p2 - b1));
    }
    tc_fence_before();
    __syncthreads();
    tc_fence_after();
    const uint32_t tmem = *s_tmem;
    // staged chunks of the CTA: all rows once for every tile, or every chunk
    // of every tile; tiles are finished in order either way
    const int nstage = nchunk > 1 ? ntile * nchunk : 1;

    int issued[2] = {0, 0};                            // (issuing thread) commits so far on each
                                                       // buffer's barrier
    if (warp == TC_WORKERS) {
        // ------------------------------------------------ MMA issue (one thread)
        if (lane == 0) {
            const uint32_t idesc = (1u << 4) | ((uint32_t)(TC_N >> 3) << 17) |
                                   ((uint32_t)(TC_M >> 4) << 24);   // M 128, N 160, fp16 K-major, fp32
            const uint32_t aZ = smem_u32(sZ);
            bool ok = true;
            for (int k = 0; k < ntile && ok; ++k) {
                // the previous tile's accumulators have been read
                if (k > 0) {
                    ok = tc_mbar_wait(bar_acc, (uint32_t)(k - 1) & 1u, limit, s_abort);
                    tc_fence_after();
                }
                for (int c = 0; c < nchunk && ok; ++c) {
                    const int i = nchunk > 1 ? k * nchunk + c : 0, b = i & (g.bufs - 1);
                    if (nchunk > 1 || k == 0)
                        ok = tc_mbar_wait(bar_full + 8 * b, (uint32_t)(i / g.bufs) & 1u, limit, s_abort);
                    if (!ok) break;
                    const uint32_t aA = smem_u32(sBuf + b * g.buf_units), aB = aA + 16u * (uint32_t)off_b;
                    const uint32_t kb = nchunk > 1 ? 0u : (uint32_t)(k * TC_N);
                    for (int t = T.n0[dir][c]; t < T.n0[dir][c + 1]; ++t) {
                        const uint4 s = sS[t];
#pragma unroll
                        for (int pa = 0; pa < 2; ++pa)
#pragma unroll
                            for (int pb = 0; pb < 2; ++pb) {
                                const uint32_t a = aA + 16u * ((uint32_t)(pa * hl_a) + s.x);
                                const uint32_t bb = aB + 16u * ((uint32_t)(pb * g.LB) + kb + s.z);
                                const uint32_t blbo = s.w == 0xffffffffu ? aZ - bb : 16u * s.w;
                                const uint32_t acc = (t > 0 || (pa == 1 && pb == 0)) ? 1u : 0u;
                                tc_mma(tmem + (uint32_t)((pa + pb) * TC_N), tc_desc(a, 16u * s.y),
                                       tc_desc(bb, blbo), idesc, acc);
                            }
                    }
                    tc_commit(bar_done + 8 * b);
                    ++issued[b];
                }
            }
            if (!ok) {
                if (!*s_abort) atomicOr(B.err[pair], (unsigned)PGM_ERR_TIMEOUT);
                *s_abort = 1;
            }
        }
        __syncwarp();
    } else {
        // ------------------------------------------------ staging and epilogue
        const int wt = tid;                            // 0 .. 255
        constexpr int WT = 32 * TC_WORKERS;
        const int o = mc.c - h;
        auto stage = [&](int tile, int c, int b) {
            uint4* sA = sBuf + b * g.buf_units;
            uint4* sB = sA + off_b;
            const int q0 = c * Q, nu = g.phases * g.LA;
            // phase slices: unit k of a slice is run q = k div pa (the last one
            // is longer), at flattened seed f = m0 + (q0 + q) Wu + j
#pragma unroll 2
            for (int e = wt; e < nu; e += WT) {
                const int ph = e / g.LA, k = e - ph * g.LA;
                const int q = min(k / g.pa, Q - 1), j = k - q * g.pa;
                const int f = m0 + (q0 + q) * g.Wu + j, v = f / g.Wu, u = f - v * g.Wu;
                const int X = sg * u + ph % sg + o, Y = sg * v + ph / sg + o;
                uint4 hi, lo;
                tc_split(tc_unit<GRAY>(D.ref, D.ref_pitch, D.rw, D.rh, X, Y, 4), hi, lo);
                sA[e] = hi;
                sA[hl_a + e] = lo;
                if (GRAY && g.copies == 2) {           // the pixels past the patch as zeros
                    tc_split(tc_unit<GRAY>(D.ref, D.ref_pitch, D.rw, D.rh, X, Y, P - tail), hi, lo);
                    sA[nu + e] = hi;
                    sA[hl_a + nu + e] = lo;
                }
            }
            // target rows: unit k is patch row r = k div pb of the chunk, at
            // flattened centre f = n0 + (r0 + r) Wt + j, pixel (f mod Wt - h, f div Wt - h)
            const int n0 = tile * TC_N, r0 = c * Q * sg, rows = min(Q * sg, P);
#pragma unroll 2
            for (int k = wt; k < g.LB; k += WT) {
                const int r = min(k / g.pb, rows - 1), j = k - r * g.pb;
                const int f = n0 + (r0 + r) * g.Wt + j, row = f / g.Wt, col = f - row * g.Wt;
                uint4 hi, lo;
                tc_split(tc_unit<GRAY>(D.tgt, D.tgt_pitch, D.tw, D.th, col - h, row - h, 4), hi, lo);
                sB[k] = hi;
                sB[g.LB + k] = lo;
            }
            // the staged operands are read by the tensor core (async proxy)
            asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
            __syncwarp();
            if (lane == 0) tc_mbar_arrive(bar_full + 8 * b);
        };
        // seed of this thread's accumulator lane
        const int quarter = warp & 3, half = warp >> 2;
        const int m = m0 + 32 * quarter + lane, si = m % g.Wu, sj = m / g.Wu;
        const bool seed_ok = si < D.nx && sj < D.ny;
        const unsigned long long sa =
            seed_ok ? D.sa2img[(size_t)(mc.c + sg * sj) * D.rw + (mc.c + sg * si)] : 0ull;
        unsigned long long best = INF;
        bool ok = true;
        // centres of a tile's columns: sum |b|^2 (INF: not a centre) and raster
        // index; two tables in turn.  A worker warp arrives on bar_tab once it
        // has written its part of tile k's table and read the whole of tile
        // k - 1's, and waits for that phase before it reads tile k's table or
        // writes tile k + 1's.  Every wait between the workers is such a
        // bounded one: a warp whose wait runs out leaves for the __syncthreads
        // at the end, and the others, which it may have left behind at any
        // point, must not wait for it without a limit.
        auto centres = [&](int k) {
            for (int j = wt; j < TC_N; j += WT) {
                const int n = (tile0 + k) * TC_N + j, y = n / g.Wt, x = n - y * g.Wt;
                const bool in = x < D.tw && y < D.th;
                const unsigned long long sb = in ? D.sb2[(size_t)y * D.sbp + x] : INF;
                sQ[(k & 1) * TC_N + j] =
                    make_uint4((uint32_t)sb, (uint32_t)(sb >> 32), (uint32_t)(y * D.tw + x), 0u);
            }
        };
        auto tables = [&](int k) {
            return __all_sync(FULL, tc_mbar_wait(bar_tab, (uint32_t)k & 1u, limit, s_abort)) != 0;
        };
        // the accumulators of tile k, complete once `waits` commits are on buffer b
        auto finish = [&](int k, int b, int waits) {
            if (!__all_sync(FULL, tc_mbar_wait(bar_done + 8 * b, (uint32_t)waits & 1u, limit, s_abort)))
                return false;
            tc_fence_after();
            const uint32_t trow = tmem + ((uint32_t)(32 * quarter) << 16);
#pragma unroll 1
            for (int c0 = 80 * half; c0 < 80 * half + 80; c0 += 16) {
                uint32_t x0[16], x1[16], x2[16];
                tc_ld16(trow + (uint32_t)c0, x0);
                tc_ld16(trow + (uint32_t)(TC_N + c0), x1);
                tc_ld16(trow + (uint32_t)(2 * TC_N + c0), x2);
#pragma unroll
                for (int j = 0; j < 16; ++j) {
                    const uint4 q = sQ[(k & 1) * TC_N + c0 + j];
                    const unsigned long long sb = (unsigned long long)q.x | ((unsigned long long)q.y << 32);
                    if (sb == INF) continue;
                    const long long cross = ((long long)__float2int_rn(__uint_as_float(x0[j])) << 14) +
                                            ((long long)__float2int_rn(__uint_as_float(x1[j])) << 7) +
                                            (long long)__float2int_rn(__uint_as_float(x2[j]));
                    const unsigned long long key = (xcost(sa, sb, cross) << 24) | q.z;
                    best = key < best ? key : best;
                }
            }
            tc_fence_before();
            __syncwarp();
            if (lane == 0) tc_mbar_arrive(bar_acc);    // accumulators free for the next tile
            return true;
        };
        if (nchunk == 1) {
            for (int k = 0; k < ntile; ++k) centres(k);
            stage(tile0, 0, 0);
            if (lane == 0) tc_mbar_arrive(bar_tab);
            ok = tables(0);
            for (int k = 0; k < ntile && ok; ++k) ok = finish(k, 0, k);
        } else {
            for (int i = 0; i <= nstage && ok; ++i) {
                const int b = i & 1, k = i / nchunk, c = i - k * nchunk;
                if (i > 0 && c == 0 && !(ok = tables(k - 1))) break;
                if (i < nstage) {
                    // the MMAs of the buffer's last chunk are done
                    if (i >= 2)
                        ok = __all_sync(FULL, tc_mbar_wait(bar_done + 8 * b, (uint32_t)(i / 2 - 1) & 1u,
                                                           limit, s_abort));
                    if (!ok) break;
                    if (c == 0) centres(k);
                    stage(tile0 + k, c, b);
                }
                if (i > 0 && c == 0)                   // the tile before is complete
                    ok = finish(k - 1, b ^ 1, (i - 1) / 2);
                if (c == 0 && ok && i < nstage && lane == 0) tc_mbar_arrive(bar_tab);
            }
        }
        if (!ok) {
            if (lane == 0) {
                if (!*s_abort) atomicOr(B.err[pair], (unsigned)PGM_ERR_TIMEOUT);
                *s_abort = 1;
            }
        }
        sBest[half * TC_M + 32 * quarter + lane] = best;
    }
    // the two column halves of a seed, then the bands of the seed
    __syncthreads();
    if (tid < TC_M && !*s_abort) {
        const unsigned long long b0 = sBest[tid], b1 = sBest[TC_M + tid];
        const unsigned long long bb = b0 < b1 ? b0 : b1;
        const int mm = m0 + tid, i = mm % g.Wu, j = mm / g.Wu;
        if (i < D.nx && j < D.ny && bb != INF) atomicMin(D.cost + (size_t)j * D.nx + i, bb);
    }
    // whichever warp gave up: the issued MMAs read shared memory and write tensor
    // memory until they finish (the last commit on each buffer is the only one
    // that can be outstanding; without an abort every one has been waited for)
    if (*s_abort && warp == TC_WORKERS && lane == 0)
        for (int b = 0; b < 2; ++b)
            if (issued[b])
                (void)tc_mbar_wait(bar_done + 8 * b, (uint32_t)(issued[b] - 1) & 1u, TC_DRAIN_CYCLES,
                                   nullptr);
    tc_fence_before();
    __syncthreads();
    if (warp == TC_WORKERS) {
        tc_fence_after();
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n"
                     ::"r"(tmem), "r"(TC_TMEM_COLS) : "memory");
    }
}

// every seed's result word starts at INF (no centre yet)
__global__ void k_init_tc_clear(const __grid_constant__ LvlBatch B) {
    const DirLvl& D = B.d[blockIdx.z][blockIdx.y];
    const int s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s < D.nx * D.ny) D.cost[s] = INF;
}

// cost << 24 | q  ->  displacement, cost and flags of every seed
__global__ void k_init_tc_fin(const __grid_constant__ LvlBatch B, const MatchConst mc) {
    const int pair = blockIdx.z, dir = blockIdx.y;
    const DirLvl& D = B.d[pair][dir];
    const int ns = D.nx * D.ny, s = blockIdx.x * blockDim.x + threadIdx.x;
    if (s == 0 && ns > 0)
        atomicAdd(B.evals[pair] + 4 + dir, (unsigned long long)ns * (unsigned long long)(D.tw * D.th));
    if (s >= ns) return;
    const unsigned long long k = D.cost[s];
    if (k == INF) {                                    // left unset (a wait ran out)
        D.u[s] = 0;
        D.flags[s] = 0;
        return;
    }
    const int q = (int)(k & 0xffffffull), si = s % D.nx, sj = s / D.nx;
    D.u[s] = pack_u(q % D.tw - (mc.c + mc.sigma * si), q / D.tw - (mc.c + mc.sigma * sj));
    D.cost[s] = k >> 24;
    D.flags[s] = F_VALID;
}

// The K steps of patch rows [ra, rb) (ra a multiple of sigma): units in raster
// order (colour: every pixel; gray: the first pixel of every run of four),
// each paired with the first later unpaired unit that also lies later in the
// staged order of the seeds (copy, phase (r mod sigma) sigma + p mod sigma,
// then r div sigma, then p div sigma), so that both operands' second offsets
// are positive; else with the zero block.  Appends to out[n ..); the new n.
int tc_pairs(int P, int sigma, bool gray, int ra, int rb, uint16_t* out, int n) {
    struct U { int p, r, key; bool used; };
    U u[TC_MAXP * TC_MAXP];
    int nu = 0;
    const int step = gray ? 4 : 1, tail = 4 * ((P - 1) / 4);
    for (int r = ra; r < rb; ++r)
        for (int p = 0; p < P; p += step) {
            const int copy = gray && P % 4 && p == tail;
            u[nu++] = {p, r,
                       (((copy * sigma + r % sigma) * sigma + p % sigma) * 64 + r / sigma) * 64 + p / sigma,
                       false};
        }
    for (int i = 0; i < nu; ++i) {
        if (u[i].used) continue;
        u[i].used = true;
        int j = i + 1;
        while (j < nu && (u[j].used || u[j].key < u[i].key)) ++j;
        if (j < nu) {
            u[j].used = true;
            out[n++] = (uint16_t)(u[i].p | u[i].r << 4 | u[j].p << 8 | u[j].r << 12);
        } else {
            out[n++] = (uint16_t)(u[i].p | u[i].r << 4 | 15 << 8 | 15 << 12);
        }
    }
    return n;
}

}  // namespace

// *handled = false (nothing launched) unless the cost is squared L2, patches
// go up to 15 x 15, and a CTA's staging fits in shared memory in chunks of at
// least sigma patch rows (sigma up to 5).  The bound is the tensor pipe: at
// the coarsest level of a dense 1024 x 436 colour pair of 3 levels (256 x 109
// seeds and centres a direction, P = 15 and 11, chunks of 5 and 6 rows) the
// kernel issues 19.3 Tflop in 13.2 ms (1.46 Pflop/s), where the per-seed
// kernel, the only other one that takes an image this wide, needs 453 ms.
// (Sixteen colour pairs of 1024 x 436, whole patches: 180 us the three launches,
// 172 before a warp of its own issued the MMAs.)
// Gray: 16 pairs of 1024 x 436 at level 4 take 87 us, against 426 us of the
// dp2a form on a staged target.
pgm_status launch_init_tc(const LvlBatch& B, const MatchConst& mc, int nch, bool* handled,
                          cudaStream_t st, int* nlaunch) {
    *handled = false;
    if (mc.norm != PGM_L2SQ || mc.sigma < 1 || B.n < 1) return PGM_OK;
    const bool gray = nch == 2;
    int units = 0, ctas = 0, seeds = 0;
    TcSteps T;
    memset(&T, 0, sizeof(T));
    for (int d = 0; d < 2; ++d) {
        const int P = B.d[0][d].P;
        for (int k = 0; k < B.n; ++k) {
            const DirLvl& D = B.d[k][d];
            if (D.P < 1 || D.P > TC_MAXP || D.P != P) return PGM_OK;
            if ((long long)D.tw * D.th >= (1ll << 24) || !D.sa2img || !D.sb2) return PGM_OK;
        }
        // the fewest chunks whose staging fits for every pair of the batch, and
        // one centre tile a CTA where more would leave SMs without one (a
        // 1024 x 436 pair had 28 CTAs with two tiles each: 1150 -> 1121 us a call,
        // a 256 x 192 gray one 474 -> 465; no gain with the line at two or four
        // CTAs a SM)
        const int nq = (P - 1) / mc.sigma + 1;
        int Q = 0, nchunk = 0, most = 0, grid = 0, per = 0;
        for (int want = 1; want <= nq && nchunk == 0; ++want) {
            Q = (nq + want - 1) / want;
            const int nc = (nq + Q - 1) / Q;
            for (per = nc > 1 ? TC_NTC : TC_NT;; per = 1) {
                int all = 0;
                most = grid = 0;
                for (int k = 0; k < B.n; ++k) {
                    const TcGeom g = tc_geom(B.d[k][d], mc.sigma, Q, nc, per, gray);
                    most = std::max(most, tc_units(g));
                    grid = std::max(grid, g.ctas);
                    all += g.ctas;
                }
                if (per == 1 || 2 * all > device_sms()) break;     // (two directions)
            }
            if (16L * most <= TC_SMEM) nchunk = nc;
        }
        if (nchunk == 0) return PGM_OK;
        T.nchunk[d] = nchunk;
        T.Q[d] = Q;
        T.per[d] = per;
        int n = 0;
        for (int c = 0; c < nchunk; ++c) {
            T.n0[d][c] = n;
            n = tc_pairs(P, mc.sigma, gray, c * Q * mc.sigma, std::min(P, (c + 1) * Q * mc.sigma),
                         T.pr[d], n);
        }
        T.n0[d][nchunk] = n;
        units = std::max(units, most);
        ctas = std::max(ctas, grid);
        for (int k = 0; k < B.n; ++k) seeds = std::max(seeds, B.d[k][d].nx * B.d[k][d].ny);
    }
    *handled = true;
    if (seeds == 0) return PGM_OK;
    const auto kern = gray ? k_init_tc<true> : k_init_tc<false>;
    if (pgm_status r = smem_opt_in((const void*)kern); r != PGM_OK) return r;
    const dim3 gs((seeds + 255) / 256, 2, B.n);
    k_init_tc_clear<<<gs, 256, 0, st>>>(B);
    kern<<<dim3(ctas, B.n, 2), TC_THREADS, 16 * units, st>>>(B, mc, T, wait_limit());
    k_init_tc_fin<<<gs, 256, 0, st>>>(B, mc);
    *nlaunch = 3;
    return launch_status("init (tensor cores): launch");
}

}  // namespace pgm
