// pm_direct.cu -- one checkerboard colour phase of propagation (Eq. 4) and
// limited random search (Eq. 5), with the cost refresh of a visit, for phases
// of few seeds (the coarse levels of a pair or a small batch), squared-L2 cost
// on int16 descriptors and either cost on the direction descriptor's
// bit-planes.
//
// Such a phase is bound by latency: there are fewer seeds than warps that the
// chip holds, and the tile kernels of pm_row.cu spend their 8 to 14 us on a
// chain of staging steps (a producer warp reads 32 seeds and places a window,
// three copies land, 14 warps score two or three seeds each).  Here every seed
// of the colour has a warp of its own that reads the seed, its neighbours and
// the patches straight from L2 (the descriptors' border of BORD pixels makes
// every patch readable without clamping), both search candidates at once.
// What is left is the launch and two or three dependent trips to L2: 4.3 us a
// colour phase of a 1024 x 436 pair at levels 4 and 3 (tiles: 10).  Within a
// trip the loads must not wait for one another: with a branch around each of a
// lane's eight loads (patches of different sizes in one code) a phase took 8 us.
// Whole visits in one launch, as a cooperative grid with barriers or as a
// cluster of 16 CTAs with the fields in shared memory, were no faster (a
// barrier of the grid costs as much as a launch, and a cluster has a tenth of
// the chip's warps).
//
// Lane l holds the pixels l, l + 32, ... of the patch in raster order; the cost
// is sum |a|^2 + sum |b|^2 - 2 sum <a, b> with dp2a on split reference bytes,
// the same exact integers as in pm_row.cu.  Bit-planes: lane r of a half-warp
// holds patch row r, a half-warp per candidate.  Candidates, order, ties and
// counts are those of pm_row.cu.
#include <limits.h>

#include "match_common.cuh"

namespace pgm {
namespace {

constexpr int PD_WARPS = 4;                  // seeds per CTA
constexpr int PD_NONE = INT_MIN;             // no propagated candidate

// the seed of a warp and what it knows before any patch is read
struct Seed {
    int s, px, py, f, f0, u, c0, c1, K;      // f: flags after the refresh, f0: as read
    bool have;
    unsigned long long cost, sa;
    uint4 r;                                 // first Philox block (search k = 0, 1)
};

template <bool BITS>
__device__ __forceinline__ Seed pd_seed(const LvlBatch& B, const MatchConst& mc, const DirLvl& D,
                                        int pair, int dir, int i, int j) {
    Seed R;
    const int t4 = mc.t & 3, sig = mc.sigma;
    const int sx = (t4 == 0 || t4 == 3) ? 1 : -1, sy = (t4 == 0 || t4 == 2) ? 1 : -1;
    const int s = j * D.nx + i, px = mc.c + sig * i, py = mc.c + sig * j;
    const int ni = i - sx, nj = j - sy;
    const bool okx = ni >= 0 && ni < D.nx, oky = nj >= 0 && nj < D.ny;
    const int sn0 = okx ? j * D.nx + ni : s, sn1 = oky ? nj * D.nx + i : s;
    const int f = D.flags[s], u = D.u[s];
    const int f0 = D.flags[sn0], f1 = D.flags[sn1], u0 = D.u[sn0], u1 = D.u[sn1];
    R.cost = D.cost[s];
    R.sa = BITS ? 0ull : D.sa2img[(size_t)py * D.rw + px];
    const int g = mc.rs_grid;                // PGM-C3/G3: level-0 search on a grid only
    R.K = mc.cost_only ? 0 : (B.level == 0 && g > 0 && !(px % g == g / 2 && py % g == g / 2)) ? 0 : mc.K;
    if (R.K > 0)
        R.r = philox(make_uint4((uint32_t)s,
                                ((uint32_t)B.visit << 16) | ((uint32_t)dir << 15) | (uint32_t)mc.t,
                                (uint32_t)B.level << 16, B.stream_id[pair]),
                     mc.key0, mc.key1);
    bool have = f & F_VALID;
    // the refresh (first iteration of a visit) drops a match whose centre left
    // the target, here and at the neighbours
    if (mc.refresh) have = have && inside(D, px + lo16((uint32_t)u), py + hi16((uint32_t)u));
    R.c0 = PD_NONE;
    R.c1 = PD_NONE;
    if (!mc.cost_only) {
        bool ok0 = okx && (f0 & F_VALID), ok1 = oky && (f1 & F_VALID);
        if (mc.refresh) {
            ok0 = ok0 && inside(D, px - sx * sig + lo16((uint32_t)u0), py + hi16((uint32_t)u0));
            ok1 = ok1 && inside(D, px + lo16((uint32_t)u1), py - sy * sig + hi16((uint32_t)u1));
        }
        // a candidate equal to the current match or to the other candidate
        // scores the same and cannot be strictly better
        if (ok0 && !(have && u0 == u) && inside(D, px + lo16((uint32_t)u0), py + hi16((uint32_t)u0)))
            R.c0 = u0;
        if (ok1 && !(ok0 && u1 == u0) && !(have && u1 == u) &&
            inside(D, px + lo16((uint32_t)u1), py + hi16((uint32_t)u1)))
            R.c1 = u1;
    }
    R.s = s; R.px = px; R.py = py; R.u = u;
    R.f0 = f;
    R.f = have ? f : (f & ~F_VALID);
    R.have = have;
    return R;
}

// search offset k of the seed (Eq. 5)
__device__ __forceinline__ void pd_offset(const LvlBatch& B, const MatchConst& mc, const Seed& R,
                                          int pair, int dir, int k, int& dx, int& dy) {
    uint4 q = R.r;
    if (k >= 2)
        q = philox(make_uint4((uint32_t)R.s,
                              ((uint32_t)B.visit << 16) | ((uint32_t)dir << 15) | (uint32_t)mc.t,
                              ((uint32_t)B.level << 16) | (uint32_t)(k >> 1), B.stream_id[pair]),
                   mc.key0, mc.key1);
    dx = rs_off((k & 1) ? q.z : q.x, k, mc.rs_W, mc.rs_mode);
    dy = rs_off((k & 1) ? q.w : q.y, k, mc.rs_W, mc.rs_mode);
}

// The candidates of one seed in the paper's order, two at a time: `cost2(c, n,
// v)` scores displacements c[0 .. n) (packed; n = 1 or 2) into v[].
template <typename Cost2>
__device__ __forceinline__ void pd_update(const LvlBatch& B, const MatchConst& mc, const DirLvl& D,
                                          const Seed& R, int pair, int dir, int lane, unsigned* cnt,
                                          Cost2 cost2) {
    bool have = R.have;
    unsigned long long bc = have && !mc.refresh ? R.cost : INF;
    int bu = R.u;
    unsigned n_eval = 0, n_cost = 0;
    // the current match (cost refresh), then the propagated ones
    int list[3];
    int n = 0;
    const bool first = mc.refresh && have;
    if (first) { list[0] = R.u; n = 1; }
    if (R.c0 != PD_NONE) { if (n == 0) list[0] = R.c0; else list[1] = R.c0; ++n; }
    if (R.c1 != PD_NONE) {
        if (n == 0) list[0] = R.c1; else if (n == 1) list[1] = R.c1; else list[2] = R.c1;
        ++n;
    }
    n_cost = first;
    n_eval = n - first;
    if (n > 0) {
        unsigned long long v[2];
        cost2(list[0], n > 1 ? list[1] : list[0], n > 1 ? 2 : 1, v);
        if (v[0] < bc) { bc = v[0]; bu = list[0]; have = true; }
        if (n > 1 && v[1] < bc) { bc = v[1]; bu = list[1]; have = true; }
        if (n > 2) {
            cost2(list[2], list[2], 1, v);
            if (v[0] < bc) { bc = v[0]; bu = list[2]; have = true; }
        }
    }
    // the limited random search around the match held after propagation
    if (have && R.K > 0) {
        const int cx = lo16((uint32_t)bu), cy = hi16((uint32_t)bu);
        for (int k = 0; k < R.K; k += 2) {
            int dx[2], dy[2], c[2];
            bool ok[2];
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                dx[e] = dy[e] = 0;
                if (k + e < R.K) pd_offset(B, mc, R, pair, dir, k + e, dx[e], dy[e]);
                ok[e] = !(dx[e] == 0 && dy[e] == 0) &&
                        inside(D, R.px + cx + dx[e], R.py + cy + dy[e]);   // tested before packing
                c[e] = pack_u(cx + dx[e], cy + dy[e]);
            }
            if (!ok[0] && !ok[1]) continue;
            unsigned long long v[2];
            const bool both = ok[0] && ok[1];
            cost2(ok[0] ? c[0] : c[1], both ? c[1] : ok[0] ? c[0] : c[1], both ? 2 : 1, v);
            n_eval += 1 + both;
            if (v[0] < bc) { bc = v[0]; bu = ok[0] ? c[0] : c[1]; }
            if (both && v[1] < bc) { bc = v[1]; bu = c[1]; }
        }
    }
    if (lane == 0) {
        if (have && (mc.refresh || bu != R.u || !(R.f & F_VALID))) {
            D.u[R.s] = bu;
            D.cost[R.s] = bc;
            D.flags[R.s] = (uint8_t)(R.f | F_VALID);
        } else if (!have && R.f != R.f0) {
            D.flags[R.s] = (uint8_t)R.f;      // the refresh dropped it
        }
        // every score is read from global memory
        atomicAdd(cnt, n_eval);
        atomicAdd(cnt + 1, n_cost);
    }
}

// int16 descriptors: lane l holds the pixels l, l + 32, ... of the P x P patch,
// M at most (4 for patches up to 11 x 11, else 8).  Every load of a patch is
// issued before the first is used: a lane's pixels past the patch read its
// corner against a zero reference word, instead of a branch around the load.
template <int M>
struct PdLane {
    unsigned rc[M];                           // row << 8 | column of pixel m (0 past the patch)
    unsigned in;                              // bit m: pixel m lies in the patch
    __device__ __forceinline__ void set(int P, int lane) {
        const unsigned inv = (65535u + (unsigned)P) / (unsigned)P;   // k / P = k inv >> 16 for k < 256
        in = 0;
#pragma unroll
        for (int m = 0; m < M; ++m) {
            const unsigned k = (unsigned)(lane + 32 * m), row = (k * inv) >> 16;
            const bool ok = (int)k < P * P;
            rc[m] = ok ? row << 8 | (k - row * (unsigned)P) : 0u;
            in |= ok ? 1u << m : 0u;
        }
    }
};

// One seed of a warp, int16 descriptors.
template <int NCH, int M>
__device__ __forceinline__ void pd_one(const LvlBatch& B, const MatchConst& mc, const PdLane<M>& L,
                                       int pair, int dir, int i, int j, int lane,
                                       unsigned* cnt) {
    constexpr int PXW = px_words(NCH), WPP = NCH / 2;
    const DirLvl& D = B.d[pair][dir];
    const int h = D.P / 2, rp = D.ref_pitch >> 1, tp = D.tgt_pitch >> 1;   // words per row
    int ra[M][WPP];
    {
        const uint32_t* img = D.ref_split + (ptrdiff_t)(mc.c + mc.sigma * j - h) * rp +
                              (ptrdiff_t)(mc.c + mc.sigma * i - h) * PXW;
        if constexpr (NCH == 6) {
            uint4 v[M];
#pragma unroll
            for (int m = 0; m < M; ++m)
                v[m] = __ldg(reinterpret_cast<const uint4*>(img + (int)(L.rc[m] >> 8) * rp + (int)(L.rc[m] & 255u) * PXW));
#pragma unroll
            for (int m = 0; m < M; ++m) {
                const bool in = (L.in >> m) & 1u;
                ra[m][0] = in ? (int)v[m].x : 0;
                ra[m][1] = in ? (int)v[m].y : 0;
                ra[m][2] = in ? (int)v[m].z : 0;
            }
        } else {
#pragma unroll
            for (int m = 0; m < M; ++m) {
                const int v = (int)__ldg(img + (int)(L.rc[m] >> 8) * rp + (int)(L.rc[m] & 255u));
                ra[m][0] = ((L.in >> m) & 1u) ? v : 0;
            }
        }
    }
    const Seed R = pd_seed<false>(B, mc, D, pair, dir, i, j);
    const uint32_t* t32 = reinterpret_cast<const uint32_t*>(D.tgt);
    auto cost2 = [&](int c0, int c1, int n, unsigned long long (&v)[2]) {
        // (n = 1: the one candidate is scored twice)
        const uint32_t* img[2];
        unsigned long long sb[2];
        int l[2] = {0, 0}, hh[2] = {0, 0};
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int c = e && n > 1 ? c1 : c0;
            int qx = R.px + lo16((uint32_t)c), qy = R.py + hi16((uint32_t)c);
            if (!PGM_CHECK(qx >= 0 && qy >= 0 && qx < D.tw && qy < D.th && h <= BORD, B.err[pair]))
                qx = qy = 0;
            sb[e] = __ldg(D.sb2 + (size_t)qy * D.sbp + qx);
            img[e] = t32 + (ptrdiff_t)(qy - h) * tp + (ptrdiff_t)(qx - h) * PXW;
        }
        if constexpr (NCH == 6) {
            uint4 w[2][M];
#pragma unroll
            for (int e = 0; e < 2; ++e)
#pragma unroll
                for (int m = 0; m < M; ++m)
                    w[e][m] = __ldg(reinterpret_cast<const uint4*>(img[e] + (int)(L.rc[m] >> 8) * tp +
                                                                   (int)(L.rc[m] & 255u) * PXW));
#pragma unroll
            for (int e = 0; e < 2; ++e)
#pragma unroll
                for (int m = 0; m < M; ++m) {
                    l[e] = __dp2a_lo((int)w[e][m].x, ra[m][0], l[e]);
                    hh[e] = __dp2a_hi((int)w[e][m].x, ra[m][0], hh[e]);
                    l[e] = __dp2a_lo((int)w[e][m].y, ra[m][1], l[e]);
                    hh[e] = __dp2a_hi((int)w[e][m].y, ra[m][1], hh[e]);
                    l[e] = __dp2a_lo((int)w[e][m].z, ra[m][2], l[e]);
                    hh[e] = __dp2a_hi((int)w[e][m].z, ra[m][2], hh[e]);
                }
        } else {
            int w[2][M];
#pragma unroll
            for (int e = 0; e < 2; ++e)
#pragma unroll
                for (int m = 0; m < M; ++m)
                    w[e][m] = (int)__ldg(img[e] + (int)(L.rc[m] >> 8) * tp + (int)(L.rc[m] & 255u));
#pragma unroll
            for (int e = 0; e < 2; ++e)
#pragma unroll
                for (int m = 0; m < M; ++m) {
                    l[e] = __dp2a_lo(w[e][m], ra[m][0], l[e]);
                    hh[e] = __dp2a_hi(w[e][m], ra[m][0], hh[e]);
                }
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) {
            const int sl = __reduce_add_sync(FULL, l[e]), sh = __reduce_add_sync(FULL, hh[e]);
            v[e] = xcost(R.sa, sb[e], (long long)sh * 128 + (long long)sl);
        }
    };
    pd_update(B, mc, D, R, pair, dir, lane, cnt, cost2);
}

// One seed of a warp, direction descriptor: popcounts on the bit-planes (see
// pm_row.cu).
template <int NCH>
__device__ __forceinline__ void pd_one_bits(const LvlBatch& B, const MatchConst& mc, int pair, int dir, int i, int j, int lane, unsigned* cnt) {
    const DirLvl& D = B.d[pair][dir];
    constexpr int NR = NCH == 6 ? 3 : 1, NW = NR + 1;   // words per row and plane: aligned, read
    const int P = D.P, h = P / 2, hf = lane >> 4, r = lane & 15;
    const unsigned fac = mc.norm == PGM_L2SQ ? 2u : 1u;
    const bool live = r < P;
    const int rr = live ? r : 0;
    unsigned msk[NR], an[NR], as[NR];
#pragma unroll
    for (int k = 0; k < NR; ++k) {
        const int nb = P * NCH - 32 * k;
        msk[k] = !live || nb <= 0 ? 0u : nb >= 32 ? 0xffffffffu : (1u << nb) - 1u;
    }
    // row rr of the patch centred at (x, y): NR aligned words of both planes
    auto row = [&](const uint32_t* bits, int brow, int height, int x, int y, unsigned (&n_)[NR],
                   unsigned (&s_)[NR]) {
        const int bit = (x - h + BORD) * NCH, sh = bit & 31;
        const uint32_t* p = bits + (size_t)(y - h + rr + BORD) * brow + (bit >> 5);
        const size_t plane = (size_t)brow * (height + 2 * BORD);
        unsigned vn[NW], vs[NW];
#pragma unroll
        for (int k = 0; k < NW; ++k) { vn[k] = __ldg(p + k); vs[k] = __ldg(p + plane + k); }
#pragma unroll
        for (int k = 0; k < NR; ++k) {
            n_[k] = __funnelshift_r(vn[k], vn[k + 1], sh);
            s_[k] = __funnelshift_r(vs[k], vs[k + 1], sh);
        }
    };
    row(D.ref_bits, D.rbit_row, D.rh, mc.c + mc.sigma * i, mc.c + mc.sigma * j, an, as);
#pragma unroll
    for (int k = 0; k < NR; ++k) an[k] &= msk[k];
    const Seed R = pd_seed<true>(B, mc, D, pair, dir, i, j);
    auto cost2 = [&](int c0, int c1, int n, unsigned long long (&v)[2]) {
        const int cu = hf && n > 1 ? c1 : c0;            // (a lone candidate is scored twice)
        const int qx = R.px + lo16((uint32_t)cu), qy = R.py + hi16((uint32_t)cu);
        unsigned c = 0;
        if (PGM_CHECK(qx >= 0 && qy >= 0 && qx < D.tw && qy < D.th && h <= BORD, B.err[pair])) {
            unsigned tn[NR], ts[NR];
            row(D.tgt_bits, D.tbit_row, D.th, qx, qy, tn, ts);
#pragma unroll
            for (int k = 0; k < NR; ++k)
                c += (unsigned)__popc((an[k] ^ tn[k]) & msk[k]) +
                     ((unsigned)__popc(an[k] & tn[k] & (as[k] ^ ts[k])) << fac);
        }
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) c += __shfl_xor_sync(FULL, c, o);
        v[0] = __shfl_sync(FULL, c, 0);
        v[1] = __shfl_sync(FULL, c, 16);
    };
    pd_update(B, mc, D, R, pair, dir, lane, cnt, cost2);
}

// One phase in a launch of its own (the refresh alone of a visit without
// iterations: both colours).
template <int NCH, bool BITS>
__global__ void __launch_bounds__(32 * PD_WARPS) k_pm_d(const __grid_constant__ LvlBatch B,
                                                        const MatchConst mc) {
    __shared__ unsigned s_cnt[2];
    pdl_trigger();
    if (threadIdx.x < 2) s_cnt[threadIdx.x] = 0u;
    __syncthreads();
    pdl_wait();
    const int dir = blockIdx.y, pair = blockIdx.z, lane = threadIdx.x & 31;
    const DirLvl& D = B.d[pair][dir];
    const int hw = (D.nx + 1) / 2, idx = (int)blockIdx.x * PD_WARPS + (int)(threadIdx.x >> 5);
    const int j = idx / hw, i = 2 * (idx - j * hw) + ((j + mc.colour) & 1);
    if (i < D.nx && j < D.ny) {
        if constexpr (BITS) {
            pd_one_bits<NCH>(B, mc, pair, dir, i, j, lane, s_cnt);
        } else if (D.P <= 11) {
            PdLane<4> L;
            L.set(D.P, lane);
            pd_one<NCH, 4>(B, mc, L, pair, dir, i, j, lane, s_cnt);
        } else {
            PdLane<8> L;
            L.set(D.P, lane);
            pd_one<NCH, 8>(B, mc, L, pair, dir, i, j, lane, s_cnt);
        }
    }
    __syncthreads();
    if (threadIdx.x < 2 && s_cnt[threadIdx.x]) {
        atomicAdd(B.evals[pair] + 2 * threadIdx.x + dir, (unsigned long long)s_cnt[threadIdx.x]);
        atomicAdd(B.evals[pair] + 6 + dir, (unsigned long long)s_cnt[threadIdx.x]);
    }
}

}  // namespace

// Seeds of one colour in the largest direction and pair of the batch, and of
// all of them together.
static void pd_sizes(const LvlBatch& B, int* most, long long* all) {
    *most = 0;
    *all = 0;
    for (int k = 0; k < B.n; ++k)
        for (int d = 0; d < 2; ++d) {
            const int n = ((B.d[k][d].nx + 1) / 2) * B.d[k][d].ny;
            *most = n > *most ? n : *most;
            *all += n;
        }
}

// The line lies where the seeds of a phase fill the chip's warps a few times
// over: 64 a SM for the colour kernel, 128 for the gray and the bit-plane
// ones, whose patches are a few loads.  Measured in us a call with the line at
// 0 (tiles only) / 16 / 32 / 64 / 128 a SM: a colour pair of 1024 x 436 1540 /
// 1289 / 1249 / 1251 / 1289, four of 1242 x 375 3184 / 3065 / 2999 / 3001 /
// 3048, one of 1920 x 1080 3512 / 3349 / 3214 / 3212 / 3271, 16 of 1024 x 436
// 9270 / 9273 / 9185 / 9161 / 9277.  Gray and bit-planes at 0 / 64 / 128 / 256:
// one 256 x 192 gray pair 737 / 488 / 487 / 489, one 640 x 480 gray direction
// pair 835 / 638 / 639 / 651, 16 direction pairs 5880 / 5769 / 5758 / 5745.
bool pm_direct_fits(const LvlBatch& B, const MatchConst& mc, int nch, int sms) {
    int most;
    long long all;
    pd_sizes(B, &most, &all);
    const int per_sm = nch == 6 && mc.descriptor != PGM_DIR ? 64 : 128;
    return all <= (long long)per_sm * sms;
}

pgm_status launch_pm_direct(const LvlBatch& B, const MatchConst& mc, int nch, cudaStream_t st) {
    int most;
    long long all;
    pd_sizes(B, &most, &all);
    if (most == 0) return PGM_OK;
    const dim3 g((most + PD_WARPS - 1) / PD_WARPS, 2, B.n);
    const bool bits = mc.descriptor == PGM_DIR;
    const auto kern = bits ? (nch == 2 ? k_pm_d<2, true> : k_pm_d<6, true>)
                           : (nch == 2 ? k_pm_d<2, false> : k_pm_d<6, false>);
    PGM_TRY(launch_pdl(kern, g, dim3(32 * PD_WARPS), 0, st, B, mc), "search: launch");
    return launch_status("search: launch");
}

}  // namespace pgm
