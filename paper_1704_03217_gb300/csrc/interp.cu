// interp.cu -- sparse-to-dense interpolation of the exported matches
// (Sec. III-G): every pixel of the reference image takes its K geodesically
// nearest matches and interpolates their displacements by a Nadaraya-Watson
// average (NW) or a locally weighted affine fit (LA), LA when the matches
// exceed 2.2 % of the image.
//
//   step cost     c(p) = 1 + (sum over descriptor channels of |g(p)|) >> shift
//   edge p - q    c(p) + c(q) on the 4-connected grid
//   neighbours    the K smallest (geodesic distance, match index) pairs
//   weights       exp(-(d - d_nearest) / lambda), in double precision
//
// The K-nearest lists are found by relaxation: a list entry (d, i) is a path
// of length d from match i, every pixel keeps its K best entries with
// distinct labels, and a pixel's candidates are its 4 neighbours' entries
// plus the step.  The fixed point is the exact K-nearest set (if match i is
// among the K nearest of p, it is among the K nearest of every pixel on a
// shortest path from i to p), and the relaxation reaches it from any order of
// updates, so the result is deterministic.  A launch relaxes 16 x 16 tiles in
// shared memory until each tile is stable; launches repeat until none
// changes anything.
//
// Every pixel carries a mask of the entries that its last round brought, and
// its neighbours look at those alone: an entry is offered once to each
// neighbour, where a list offered whole whenever anything in it changed cost
// most of its comparisons on entries already refused.  A launch works on the
// tiles next to one that changed in the launch before, from their halo
// inwards.  The bound is the integer ALU pipe (86 % busy at 1024 x 436, 16
// neighbours, matches at three fifths of a grid of 3): the list insertions.
// Times: see pgm_interpolate.
#include <stdint.h>

#include "pgm_device.cuh"

namespace pgm {
namespace {

constexpr int IT_W = 16;                 // tile side (pixels), one thread each
constexpr int IT_H = IT_W + 2;           // with the 1-pixel halo
constexpr int IK_MAX = 16;               // neighbours per pixel at most
// relaxation rounds per launch and tile: few, so that entries from the next
// tile come before a tile has settled without them (1024 x 436, ms a call at 2,
// 3, 4, 6, 8, 12 rounds: 3.18, 2.98, 3.01, 3.07, 3.19, 3.46)
constexpr int IT_INNER = 4;
constexpr unsigned long long EMPTY = ~0ull;

// key = distance << 32 | match index; ascending keys are the (d, i) order
__device__ __forceinline__ unsigned lab_of(unsigned long long k) { return (unsigned)k; }

// Insert a candidate that is below the k-th entry into a sorted list of k
// distinct labels: an entry of the same label that is no worse keeps it out, a
// worse one (else the last) gives way.  Bit e of `fresh` belongs to entry e and
// moves with it; the candidate's is set.
__device__ __forceinline__ void list_insert(unsigned long long (&L)[IK_MAX], unsigned& fresh, int k,
                                            unsigned long long cand) {
    const unsigned lab = lab_of(cand);
    int pos = 0, out = k - 1;                 // its place; the entry that leaves
    bool same = false;
#pragma unroll
    for (int e = 0; e < IK_MAX; ++e) {
        pos += L[e] <= cand;
        if (lab_of(L[e]) == lab) { out = e; same = true; }     // (an empty entry's label is no index)
    }
    if (same && out < pos) return;
#pragma unroll
    for (int e = IK_MAX - 1; e >= 0; --e) {
        if (e > 0 && e > pos && e <= out) L[e] = L[e > 0 ? e - 1 : 0];
        if (e == pos) L[e] = cand;
    }
    const unsigned low = (1u << pos) - 1u, mid = ((1u << out) - 1u) & ~low;
    fresh = (fresh & low) | ((fresh & mid) << 1) | (1u << pos) | (fresh & ~((2u << out) - 1u));
}

// step costs, empty lists, and the weights exp(-d / lambda) of the distances d
// below IW_TAB (k_iflow: an exponential in double precision per neighbour was
// most of its time)
constexpr int IW_TAB = 4096;
__global__ void k_icost(const int16_t* desc, int row, int pxe, int nch, int w, int h, int shift,
                        int k, double lambda, uint32_t* cost, unsigned long long* keys, double* tab) {
    const int64_t n = (int64_t)w * h, first = (int64_t)blockIdx.x * blockDim.x, p = first + threadIdx.x;
    for (int64_t i = p; i < IW_TAB; i += (int64_t)gridDim.x * blockDim.x) tab[i] = exp(-(double)i / lambda);
    for (int e = 0; e < k; ++e) {             // the block's lists, one after another
        const int64_t i = first * k + (int64_t)e * blockDim.x + threadIdx.x;
        if (i < n * k) keys[i] = EMPTY;
    }
    if (p >= n) return;
    const int x = (int)(p % w), y = (int)(p / w);
    const int16_t* g = desc + (int64_t)y * row + (int64_t)x * pxe;
    long long s = 0;
    for (int c = 0; c < nch; ++c) s += g[c] < 0 ? -(int)g[c] : (int)g[c];
    cost[p] = 1u + (uint32_t)(s >> shift);
}

// every match enters its pixel's list at distance 0 (the smaller index where
// two share a pixel)
__global__ void k_iseed(const int32_t* rows, const int32_t* count, int64_t max_rows, int w, int h,
                        int k, unsigned long long* keys) {
    const int64_t n = min((int64_t)*count, max_rows);
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int x = rows[4 * i], y = rows[4 * i + 1];
        if (x < 0 || y < 0 || x >= w || y >= h) continue;
        atomicMin(keys + ((int64_t)y * w + x) * k, (unsigned long long)i);
    }
}

// Tile states after a launch: unchanged, changed, and not yet stable when the
// launch's rounds ran out.
enum { TILE_SAME = 0, TILE_CHANGED = 1, TILE_OPEN = 2 };
constexpr int IL = IK_MAX + 1;                // keys per staged list: neighbouring pixels' entries in
                                              // different banks

// KT > 0: k fixed at compile time (16, the default, and 8); KT = 0: any k.  was: tile
// states of the launch before (null: the first launch); now: of this one; open
// tiles leave the entries of their last round in `left` and go on from there.
// prev: whether the launch before changed anything (null: not to be asked).
template <int KT>
__global__ void __launch_bounds__(IT_W * IT_W) k_irelax(const uint32_t* cost, int w, int h, int k_,
                                                        unsigned long long* keys, const uint8_t* was,
                                                        uint8_t* now, uint16_t* left,
                                                        const unsigned* prev, unsigned* changed) {
    if (prev && *prev == 0u) return;
    const int k = KT > 0 ? KT : k_;
    __shared__ unsigned long long sl[IT_H * IT_H][IL];
    __shared__ uint32_t sc[IT_H * IT_H];
    __shared__ uint16_t fresh[2][IT_H * IT_H];    // entries that the last round brought
    const int tile = blockIdx.y * gridDim.x + blockIdx.x;
    int self = TILE_OPEN, nl = 1, nr = 1, nu = 1, nd = 1;      // own state, neighbours changed
    if (was) {
        self = was[tile];
        nl = blockIdx.x > 0 && was[tile - 1] != TILE_SAME;
        nr = blockIdx.x + 1 < gridDim.x && was[tile + 1] != TILE_SAME;
        nu = blockIdx.y > 0 && was[tile - (int)gridDim.x] != TILE_SAME;
        nd = blockIdx.y + 1 < gridDim.y && was[tile + (int)gridDim.x] != TILE_SAME;
        if (self != TILE_OPEN && !(nl | nr | nu | nd)) {       // (uniform)
            if (threadIdx.x == 0) now[tile] = TILE_SAME;
            return;
        }
    }
    const int tx = threadIdx.x % IT_W, ty = threadIdx.x / IT_W;
    const int x0 = blockIdx.x * IT_W - 1, y0 = blockIdx.y * IT_W - 1;
    for (int i = threadIdx.x; i < IT_H * IT_H * IK_MAX; i += IT_W * IT_W) {
        const int t = i / IK_MAX, e = i % IK_MAX, x = x0 + t % IT_H, y = y0 + t / IT_H;
        const bool in = x >= 0 && y >= 0 && x < w && y < h;
        sl[t][e] = in && e < k ? keys[((int64_t)y * w + x) * k + e] : EMPTY;
    }
    for (int t = threadIdx.x; t < IT_H * IT_H; t += IT_W * IT_W) {
        const int cx = t % IT_H, cy = t / IT_H, x = x0 + cx, y = y0 + cy;
        sc[t] = x >= 0 && y >= 0 && x < w && y < h ? cost[(int64_t)y * w + x] : 0u;
        // round 0 looks at the neighbouring tiles' edges where those changed
        // (which of the entries are new is not known: they may be changing
        // now), and at what an open tile's last round left
        const bool inner = cx > 0 && cx < IT_H - 1 && cy > 0 && cy < IT_H - 1;
        const bool f = cx == 0 ? nl : cx == IT_H - 1 ? nr : cy == 0 ? nu : cy == IT_H - 1 ? nd : !was;
        fresh[0][t] = f ? 0xffffu : inner && self == TILE_OPEN && sc[t] ? left[(int64_t)y * w + x] : 0u;
        fresh[1][t] = 0;
    }
    __syncthreads();
    const int x = x0 + 1 + tx, y = y0 + 1 + ty, me = (ty + 1) * IT_H + tx + 1;
    const bool live = x < w && y < h;
    unsigned long long L[IK_MAX];
#pragma unroll
    for (int e = 0; e < IK_MAX; ++e) L[e] = sl[me][e];
    bool any = false, open = true;
    unsigned ch = 0;
    for (int it = 0; it < IT_INNER; ++it) {
        ch = 0;
        const int cur = it & 1;
        if (live) {
            const int nb[4] = {me - 1, me + 1, me - IT_H, me + IT_H};
#pragma unroll 1
            for (int q = 0; q < 4; ++q) {
                const int t = q == 0 ? nb[0] : q == 1 ? nb[1] : q == 2 ? nb[2] : nb[3];
                unsigned m = fresh[cur][t];
                if (sc[t] == 0u) m = 0;                          // outside the image
                const unsigned step = sc[me] + sc[t];
                while (m) {
                    const unsigned long long key = sl[t][__ffs(m) - 1];
                    m &= m - 1;
                    if (key == EMPTY) break;
                    if ((key >> 32) + step >= 0xffffffffull) break;   // out of range
                    const unsigned long long cand = key + ((unsigned long long)step << 32);
                    // no better than the worst entry: neither are the larger
                    // ones after it
                    unsigned long long worst = EMPTY;
#pragma unroll
                    for (int f = 0; f < IK_MAX; ++f)
                        if (f == k - 1) worst = L[f];
                    if (cand >= worst) break;
                    list_insert(L, ch, k, cand);
                }
            }
        }
        __syncthreads();                                         // everyone has read
        if (ch) {
#pragma unroll
            for (int e = 0; e < IK_MAX; ++e) sl[me][e] = L[e];
        }
        fresh[cur ^ 1][me] = (uint16_t)ch;                       // read in the next round
        if (threadIdx.x < 4 * IT_H) {                            // the halo does not change
            const int e = threadIdx.x, t = e < IT_H ? e : e < 2 * IT_H ? (IT_H - 1) * IT_H + e - IT_H
                                              : e < 3 * IT_H ? (e - 2 * IT_H) * IT_H
                                                             : (e - 3 * IT_H) * IT_H + IT_H - 1;
            fresh[cur ^ 1][t] = 0;
        }
        any |= ch != 0;
        if (!__syncthreads_or(ch != 0)) { open = false; break; }   // the tile is stable
    }
    if (live && any) {
        const int64_t p = (int64_t)y * w + x;
#pragma unroll
        for (int e = 0; e < IK_MAX; ++e)
            if (e < k) keys[p * k + e] = L[e];
    }
    if (live && open) left[(int64_t)y * w + x] = (uint16_t)ch;
    if (__syncthreads_or(any)) {
        if (threadIdx.x == 0) {
            now[tile] = open ? TILE_OPEN : TILE_CHANGED;
            atomicOr(changed, 1u);
        }
    } else if (threadIdx.x == 0) {
        now[tile] = TILE_SAME;
    }
}

// NW or LA at every pixel; double precision without contraction, in the
// order of the plain definition
// (products with the constant 1 left out, equal sums kept once: the same bits
// with half the operations; the bound is the double-precision rate)
__global__ void k_iflow(const unsigned long long* keys, int w, int h, int k, const int32_t* rows,
                        const int32_t* count, int64_t max_rows, int mode, int permyriad,
                        double lambda, const double* tab, float* flow) {
    const int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (p >= (int64_t)w * h) return;
    const int64_t n = min((int64_t)*count, max_rows);
    const bool use_la = mode == PGM_INTERP_LA ||
                        (mode == PGM_INTERP_AUTO && n * 10000 > (int64_t)permyriad * w * h);
    const int x = (int)(p % w), y = (int)(p / w);
    double sw = 0, nwx = 0, nwy = 0;
    double m00 = 0, m01 = 0, m10 = 0, m11 = 0, m02 = 0, m12 = 0;
    double bx0 = 0, bx1 = 0, by0 = 0, by1 = 0;
    const unsigned long long d0 = keys[p * k] >> 32;
    for (int e = 0; e < k; ++e) {
        const unsigned long long key = keys[p * k + e];
        if (key == EMPTY) break;
        const int64_t i = (int64_t)(key & 0xffffffffu);
        const unsigned long long d = (key >> 32) - d0;
        const double wgt = d < (unsigned long long)IW_TAB ? tab[d] : exp(-(double)d / lambda);
        const int sx = rows[4 * i], sy = rows[4 * i + 1];
        const double wfx = __dmul_rn(wgt, (double)(rows[4 * i + 2] - sx));
        const double wfy = __dmul_rn(wgt, (double)(rows[4 * i + 3] - sy));
        sw = __dadd_rn(sw, wgt);
        nwx = __dadd_rn(nwx, wfx);
        nwy = __dadd_rn(nwy, wfy);
        if (use_la) {
            const double v0 = (double)(sx - x), v1 = (double)(sy - y);
            const double w0 = __dmul_rn(wgt, v0), w1 = __dmul_rn(wgt, v1);
            m00 = __dadd_rn(m00, __dmul_rn(w0, v0));
            m01 = __dadd_rn(m01, __dmul_rn(w0, v1));
            m10 = __dadd_rn(m10, __dmul_rn(w1, v0));
            m11 = __dadd_rn(m11, __dmul_rn(w1, v1));
            m02 = __dadd_rn(m02, w0);
            m12 = __dadd_rn(m12, w1);
            bx0 = __dadd_rn(bx0, __dmul_rn(wfx, v0));
            bx1 = __dadd_rn(bx1, __dmul_rn(wfx, v1));
            by0 = __dadd_rn(by0, __dmul_rn(wfy, v0));
            by1 = __dadd_rn(by1, __dmul_rn(wfy, v1));
        }
    }
    const double M[3][3] = {{m00, m01, m02}, {m10, m11, m12}, {m02, m12, sw}};
    const double bx[3] = {bx0, bx1, nwx}, by[3] = {by0, by1, nwy};
    double ox = 0, oy = 0;
    if (sw > 0) {
        ox = nwx / sw;
        oy = nwy / sw;
        if (use_la) {
            auto mul = [](double a, double b) { return __dmul_rn(a, b); };
            auto sub = [](double a, double b) { return __dsub_rn(a, b); };
            auto add = [](double a, double b) { return __dadd_rn(a, b); };
            const double det = add(sub(mul(M[0][0], sub(mul(M[1][1], M[2][2]), mul(M[1][2], M[2][1]))),
                                       mul(M[0][1], sub(mul(M[1][0], M[2][2]), mul(M[1][2], M[2][0])))),
                                   mul(M[0][2], sub(mul(M[1][0], M[2][1]), mul(M[1][1], M[2][0]))));
            if (det > mul(mul(mul(1e-6, sw), sw), sw)) {
                const double dx = add(sub(mul(M[0][0], sub(mul(M[1][1], bx[2]), mul(bx[1], M[2][1]))),
                                          mul(M[0][1], sub(mul(M[1][0], bx[2]), mul(bx[1], M[2][0])))),
                                      mul(bx[0], sub(mul(M[1][0], M[2][1]), mul(M[1][1], M[2][0]))));
                const double dy = add(sub(mul(M[0][0], sub(mul(M[1][1], by[2]), mul(by[1], M[2][1]))),
                                          mul(M[0][1], sub(mul(M[1][0], by[2]), mul(by[1], M[2][0])))),
                                      mul(by[0], sub(mul(M[1][0], M[2][1]), mul(M[1][1], M[2][0]))));
                ox = dx / det;
                oy = dy / det;
            }
        }
    }
    flow[2 * p] = (float)ox;
    flow[2 * p + 1] = (float)oy;
}

}  // namespace

// workspace: the lists (w h k keys), the step costs, the change flags, the
// weights, two sets of tile states and what open tiles' last rounds left
constexpr int IR_GROUP = 8;                   // relaxation launches between two looks at the flags
struct IPlan { size_t off_keys, off_cost, off_flag, off_tab, off_tile[2], off_left, bytes; int tx, ty; };
static bool make_iplan(int w, int h, int k, IPlan* ip) {
    if (w < 1 || h < 1 || w > 32767 || h > 32767 || k < 1 || k > IK_MAX) return false;
    auto al = [](size_t v) { return (v + 255) & ~(size_t)255; };
    const size_t n = (size_t)w * h;
    ip->tx = (w + IT_W - 1) / IT_W;
    ip->ty = (h + IT_W - 1) / IT_W;
    ip->off_keys = 0;
    ip->off_cost = al(n * k * 8);
    ip->off_flag = ip->off_cost + al(n * 4);
    ip->off_tab = ip->off_flag + 256;
    ip->off_tile[0] = ip->off_tab + al(IW_TAB * 8);
    ip->off_tile[1] = ip->off_tile[0] + al((size_t)ip->tx * ip->ty);
    ip->off_left = ip->off_tile[1] + al((size_t)ip->tx * ip->ty);
    ip->bytes = ip->off_left + al(n * 2);
    return true;
}

}  // namespace pgm

using namespace pgm;

extern "C" {

void pgm_interp_default_params(pgm_interp_params* ip) {
    if (!ip) return;
    ip->k = 16;
    ip->mode = PGM_INTERP_AUTO;
    ip->cost_shift = 10;
    ip->la_permyriad = 220;
    ip->lambda = 32.0;
}

size_t pgm_interp_workspace_bytes(int w, int h, const pgm_interp_params* ip) {
    IPlan pl;
    return ip && make_iplan(w, h, ip->k, &pl) ? pl.bytes : 0;
}

pgm_status pgm_interpolate(const pgm_params* p, const void* d_pyr1, int w, int h,
                           const int32_t* d_matches, const int32_t* d_count, int64_t max_matches,
                           const pgm_interp_params* ip, void* d_ws, size_t ws_bytes,
                           float* d_flow, void* stream) {
    pgm_status r = check_params(p);
    if (r != PGM_OK) return r;
    if (!ip || !d_pyr1 || !d_count || !d_ws || !d_flow || max_matches < 0 ||
        (max_matches > 0 && !d_matches) || ip->cost_shift < 0 || ip->cost_shift > 31 ||
        !(ip->lambda > 0) || ip->la_permyriad < 0 || ip->mode < PGM_INTERP_AUTO ||
        ip->mode > PGM_INTERP_LA || (((uintptr_t)d_ws) & 255u))
        return PGM_ERR_ARG;
    PyrPlan pp;
    IPlan pl;
    if (!make_pyr_plan(p, w, h, &pp) || !make_iplan(w, h, ip->k, &pl)) return PGM_ERR_ARG;
    if (ws_bytes < pl.bytes) return PGM_ERR_WORKSPACE;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    uint8_t* ws = static_cast<uint8_t*>(d_ws);
    auto* keys = reinterpret_cast<unsigned long long*>(ws + pl.off_keys);
    auto* cost = reinterpret_cast<uint32_t*>(ws + pl.off_cost);
    auto* flag = reinterpret_cast<unsigned*>(ws + pl.off_flag);
    auto* tab = reinterpret_cast<double*>(ws + pl.off_tab);
    auto* left = reinterpret_cast<uint16_t*>(ws + pl.off_left);
    const int16_t* desc = reinterpret_cast<const int16_t*>(static_cast<const uint8_t*>(d_pyr1) +
                                                           pp.desc_off[0][0]);
    Range range("pgm_interpolate");
    const int64_t n = (int64_t)w * h;
    const int blocks = (int)((n + 255) / 256);
    k_icost<<<blocks, 256, 0, st>>>(desc, pp.desc_row[0], 2 * pp.pxw, pp.nch, w, h, ip->cost_shift,
                                    ip->k, ip->lambda, cost, keys, tab);
    if ((r = launch_status("interpolate: costs")) != PGM_OK) return r;
    if (max_matches > 0) {
        k_iseed<<<152, 256, 0, st>>>(d_matches, d_count, max_matches, w, h, ip->k, keys);
        if ((r = launch_status("interpolate: seeds")) != PGM_OK) return r;
    }
    // relax until a launch changes nothing, in groups of launches between two
    // looks at their flags (a launch after one that changed nothing returns at
    // once).  The bound keeps a defect from looping for ever: a launch carries
    // the entries at least one pixel further on their shortest paths (IT_INNER
    // pixels inside a tile, one where a path crosses between two tiles at every
    // step; one launch more where a neighbour's list was being written while it
    // was read), and a path has at most w h pixels.  1024 x 436, k = 16, LA: the
    // call 12.1 -> 3.0 ms (relaxation 11.6 -> 2.5 in 16 launches, interpolation
    // 1.0 -> 0.47).
    const dim3 grid(pl.tx, pl.ty);
    const long long most = 4ll * (long long)w * h + 64;
    long long launches = 0;
    for (bool more = true; more;) {
        if (launches > most) return PGM_ERR_UNSUPPORTED;
        PGM_TRY(cudaMemsetAsync(flag, 0, 4 * IR_GROUP, st), "interpolate: clear the flags");
        for (int g = 0; g < IR_GROUP; ++g, ++launches) {
            const uint8_t* was = launches ? ws + pl.off_tile[(launches + 1) & 1] : nullptr;
            uint8_t* now = ws + pl.off_tile[launches & 1];
            const unsigned* prev = g ? flag + g - 1 : nullptr;
            const auto kern = ip->k == IK_MAX ? k_irelax<IK_MAX> : ip->k == 8 ? k_irelax<8> : k_irelax<0>;
            kern<<<grid, IT_W * IT_W, 0, st>>>(cost, w, h, ip->k, keys, was, now, left, prev, flag + g);
        }
        if ((r = launch_status("interpolate: relax")) != PGM_OK) return r;
        unsigned host_flag[IR_GROUP];
        PGM_TRY(cudaMemcpyAsync(host_flag, flag, 4 * IR_GROUP, cudaMemcpyDeviceToHost, st),
                "interpolate: read the flags");
        PGM_TRY(cudaStreamSynchronize(st), "interpolate: synchronize");
        for (int g = 0; g < IR_GROUP; ++g) more = more && host_flag[g] != 0;
    }
    k_iflow<<<blocks, 256, 0, st>>>(keys, w, h, ip->k, d_matches, d_count, max_matches, ip->mode,
                                    ip->la_permyriad, ip->lambda, tab, d_flow);
    return launch_status("interpolate: flow");
}

}  // extern "C"
