// lbs_solve2.cuh — the Crank-Nicolson solve of a 2D step (arXiv 2311.15242,
// Sec. 2.2) with the whole grid resident on the chip: colour gradient and
// weights at t+1, every red-black SOR sweep, the conserved total and the
// rescale in one launch, in FP32 arithmetic.
//
// The grid is cut into tiles, one a block, at most one block an SM, all
// running at once (a cooperative launch; a batch runs several grids, each by
// its own gang of blocks, see lbs_batch.cu).  A block keeps its tile and a
// halo of H cells (a region of at most 64 x 64) in registers: lane l of warp w
// holds the cell pairs 2 l, 2 l + 1 of the rows 4 w .. 4 w + 3: psi, C, and the
// faces and inverse diagonals of their rows (the right-hand sides wait in shared
// memory for want of registers).  An update is that of sor_tile2_cb, operation by
// operation and rounding by rounding, so the results are its own to the bit
// (but where the totals, summed in other orders, differ by an ulp and a cell's
// rescale rounds apart: once in about 3 10^8 cells times steps).  The x-neighbour outside the pair comes from the
// adjacent lane by shuffle; of the y-neighbours only those in another warp's rows
// go through shared memory.  A half-sweep
// updates one cell of every pair, spreads the error of the stale region edge
// by one cell, and ends with a block barrier.
//
// NR rounds of K sweeps (H = 2 K NR) run between two grid barriers.  A round
// is what the convergence test looks at (lbs_set_sor_tile's sweeps a round),
// so the state after every round is kept (in shared memory) until the test has been
// made: the result is that of the first round that meets the tolerance, and
// does not depend on NR.
//
// What bounds it: latency, a chain of some 35 block barriers and two grid
// barriers with L2 round trips, and the fetching of its instructions.  At 256 x
// 1024 (8 sweeps, FP32) k_sorfuse2 (32 x 16 tiles, 2 sweeps a round: twelve 8-byte
// shared accesses and about 60 instructions an update, FP64 in every thread's
// reductions, a grid barrier of 512 blocks five times) takes 65 us, this form
// 34 with 145 blocks (about 9 until the first sweep, 2 x 4.4 for 4 sweeps, 2 x 5
// from publishing the tile to the decision; 36 % of the issue slots); at 64 x 517
// (33 blocks, 6 sweeps) 53 -> 33 us, at 241 x 1011 (odd periodic axis) 90 -> 41.
#pragma once

#include <type_traits>

#include "lbs_k2d.cuh"

namespace lbs {

// tiles of an nx x ny grid: along an axis of n cells the tile boundaries are
// 0, e + t, e + 2 t, ..., n (t even; e = H where the axis ends at walls or
// mirror planes, whose outermost tiles need no halo beyond them, else 0)
struct SolveGeom {
    int ntx, nty;  // tiles
    int tx, ty;    // t along x and y
    int ex, ey;    // e along x and y
};

constexpr int kSolveRegion = 64;   // largest side of a region
constexpr int kSolveThreads = 512;
constexpr int kSolveMaxBlocks = 256;  // blocks of a gang at most
constexpr int kSolveFine = 32;        // blocks from which a warp's sums are pairs

// what a block leaves for the others at a grid barrier: for each of at most
// two rounds the largest |d psi|, |d C|, |psi|, |C| of its last sweep and the
// surfactant sum of the tile
struct __align__(16) SolveRec {
    float m[8];
    double2 sum;  // of the two rounds
};
constexpr size_t kSolveRecBytes = 2 * (size_t)kSolveMaxBlocks * sizeof(SolveRec);

// tile side and number of tiles along an axis: n cells, `walled` ends, halo H,
// regions of at most `region` cells, at most `most` tiles; the smallest number of tiles >= least that fits the
// region; false if none does
inline bool solve_axis(int n, bool walled, int H, int region, int least, int most, int &nt, int &t,
                       int &e) {
    e = walled ? H : 0;
    const int inner = region - 2 * H;
    for (int want = least < 1 ? 1 : least; want <= most; want++) {
        const int m = n - 2 * e;
        nt = want;
        t = m > 0 ? (m + nt - 1) / nt : 2;
        t += t & 1;
        while (nt > 1 && e + (nt - 1) * t >= n) nt--;  // (rounding up left a tile empty)
        if (nt == 1) {
            t = n + (n & 1);
            if (walled ? n <= region : t <= inner) return true;
        } else if (t <= inner && n - e - (nt - 1) * t <= inner + (walled ? H : 0)) {
            return true;
        }
    }
    return false;
}

// a grid of at most `blocks` tiles for halo H, or false: as few columns of
// tiles as fit (a row of a tile costs its 64 lanes whatever its width);
// rows: `small` asks for tiles as flat as 16 rows, spread over more blocks
// (shorter when the launch has the chip to itself), else for as few as fit
inline bool solve_geom(int nx, int ny, const int *wall, int H, int blocks, bool small,
                       SolveGeom &g) {
    if (blocks > kSolveMaxBlocks) blocks = kSolveMaxBlocks;
    if (!solve_axis(nx, wall[0] != 0, H, kSolveRegion, 1, blocks, g.ntx, g.tx, g.ex)) return false;
    const int most = blocks / g.ntx;
    int least = 1;
    if (small) {
        least = (ny + 15) / 16;
        if (least > most) least = most;
    }
    return solve_axis(ny, wall[1] != 0, H, kSolveRegion, least, most, g.nty, g.ty, g.ey) &&
           (long long)g.ntx * g.nty <= blocks;
}

template <int NR>
struct SolveSmem {
    static constexpr int N = kSolveRegion;
    // weights and right-hand sides of the region; rows of psi, C that
    // other warps read; the kept round's psi, C (NR > 1): all [row][column parity][column / 2], so that a
    // warp's accesses are consecutive.  The colour fractions of the region and
    // the ring around it, needed before the sweeps only, share the space of the
    // latter two: rows -1 .. N, columns -2 .. N + 1.
    static constexpr int FS = N / 2 + 2;  // columns of one parity
    static constexpr size_t w_bytes = (size_t)N * N * sizeof(float2);
    static constexpr size_t x_bytes = (size_t)N * N * sizeof(float2);
    static constexpr size_t f_bytes = (size_t)(N + 2) * 2 * FS * sizeof(float2);
    static constexpr size_t snap_bytes = NR > 1 ? x_bytes : 0;
    static constexpr size_t bytes =
        2 * w_bytes + (x_bytes + snap_bytes > f_bytes ? x_bytes + snap_bytes : f_bytes);
};

// (scalar operations: the packed ones of sm_103a, add / mul / fma.f32x2, have the
// throughput of two scalar ones; here they brought nothing)
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) {
    return make_float2(fmaf(a.x, b.x, c.x), fmaf(a.y, b.y, c.y));
}
__device__ __forceinline__ float2 shfl_up2(float2 v) {
    return make_float2(__shfl_up_sync(0xffffffffu, v.x, 1), __shfl_up_sync(0xffffffffu, v.y, 1));
}
__device__ __forceinline__ float2 shfl_down2(float2 v) {
    return make_float2(__shfl_down_sync(0xffffffffu, v.x, 1), __shfl_down_sync(0xffffffffu, v.y, 1));
}
// largest of a warp's non-negative floats
__device__ __forceinline__ float warp_max_pos(float v) {
    return __uint_as_float(__reduce_max_sync(0xffffffffu, __float_as_uint(v)));
}
// a sum as three floats, hi + lo + rest: adding another keeps the rounding errors
// of hi and of lo, so that some 70 bits count
__device__ __forceinline__ void add3(float &hi, float &lo, float &rest, float h, float l, float r) {
    float e, el, ee;
    hi = two_sum(hi, h, e);
    lo = two_sum(two_sum(lo, l, el), e, ee);
    rest = (rest + r) + (el + ee);
}
// the sums of groups of 2 `from` lanes, of NR rounds side by side, in every lane; not
// `fine`: as pairs (48 bits)
template <int NR>
__device__ __forceinline__ void lane_sum3(float (&hi)[NR], float (&lo)[NR], float (&rest)[NR],
                                          bool fine, int from = 16) {
    if (!fine) {
#pragma unroll
        for (int n = 0; n < NR; n++) {
            lo[n] += rest[n];
            rest[n] = 0.f;
        }
#pragma unroll 1
        for (int o = 16; o > 0; o >>= 1) {
            float h[NR], l[NR], e;
#pragma unroll
            for (int n = 0; n < NR; n++) {
                h[n] = __shfl_xor_sync(0xffffffffu, hi[n], o);
                l[n] = __shfl_xor_sync(0xffffffffu, lo[n], o);
            }
#pragma unroll
            for (int n = 0; n < NR; n++) {
                hi[n] = two_sum(hi[n], h[n], e);
                lo[n] = (lo[n] + l[n]) + e;
            }
        }
        return;
    }
#pragma unroll 1
    for (int o = from; o > 0; o >>= 1) {
        float h[NR], l[NR], r[NR];
#pragma unroll
        for (int n = 0; n < NR; n++) {
            h[n] = __shfl_xor_sync(0xffffffffu, hi[n], o);
            l[n] = __shfl_xor_sync(0xffffffffu, lo[n], o);
            r[n] = __shfl_xor_sync(0xffffffffu, rest[n], o);
        }
#pragma unroll
        for (int n = 0; n < NR; n++) add3(hi[n], lo[n], rest[n], h[n], l[n], r[n]);
    }
}
// a plane's element at a byte offset (32 bits: one register an address)
__device__ __forceinline__ float &at(float *p, unsigned o) { return *(float *)((char *)p + o); }

// d <= tol x, the product not rounded (as in double precision)
__device__ __forceinline__ bool at_most(float d, float tol, float x) {
    const float p = __fmul_rn(tol, x);
    return d < p || (d == p && !(fmaf(tol, x, -p) < 0.f));
}
// the decision of round_converged from the maxima themselves (m: |d psi|,
// |d C|, |psi|, |C|; before: the largest update of the round before)
__device__ __forceinline__ bool solve_converged(const float *m, float before, bool first,
                                                float tol) {
    if (at_most(m[0], tol, m[2]) && at_most(m[1], tol, m[3])) return true;
    if (first || !(at_most(m[0], 8.f * tol, m[2]) && at_most(m[1], 8.f * tol, m[3]))) return false;
    return fmaxf(m[0], m[1]) >= 0.5f * before;
}

// tile (bx, by), block `blk` of the nb of grid I's gang.  FP64 runs at 1/64 of
// FP32's rate, so the surfactant is summed in compensated FP32 pairs within a
// thread (8 cells) and a warp (256; their errors average out over the warps, but
// a gang of fewer than 32 blocks takes three floats a sum: of 11 warps, pairs
// were off by four times FP64's error), in three floats across a block's warps (a
// chain of FP64 adds there costs a step 1 us) and in FP64 across the blocks, once,
// when the round that ends the solve is known.  The code is kept short (loops over
// a thread's cells are rolled where the cells can pass through shared memory): with
// little work a thread, the time of a launch is that of fetching its
// instructions; unrolled over the eight cells it had 144 KB of code and took
// 47 us at 256 x 1024.
template <int K, int NR>
__device__ __forceinline__ void solve2_tile(const Inst<float> &I, const SolveGeom &g, int bx,
                                            int by, int blk, int nb, int max_rounds,
                                            long long max_looks, unsigned char *smem) {
    constexpr int N = kSolveRegion, H = 2 * K * NR, NW = kSolveThreads / 32;
    using S = SolveSmem<NR>;
    constexpr int FS = S::FS;
    float2 *Ws = (float2 *)smem;
    float2 *Bs = (float2 *)(smem + S::w_bytes);
    float2 *Xs = (float2 *)(smem + 2 * S::w_bytes);
    float2 *Fr = Xs;
    float2 *Sn = (float2 *)(smem + 2 * S::w_bytes + S::x_bytes);
    __shared__ __align__(16) float redm[NW][8], redb[8][8];
    __shared__ float strip[3][kSolveThreads];  // the threads' sums of the first round of two
    __shared__ float reds[3][2][NW];           // the warps' sums of the rounds
    __shared__ double2 sums[kSolveMaxBlocks];  // the blocks' sums of the last phase
    __shared__ struct {
        double M0;     // the conserved total
        float dscale;  // rescale step
        int ok;        // the barrier's wait ended well
    } st;
    __shared__ uint4 offs[kSolveThreads];
    const int tid = threadIdx.x, l = tid & 31, w = tid >> 5;
    Ctl *ctl = I.ctl;
    const long long step0 = ctl->step;  // (block 0 advances it at the end)
    const MomSet<float> m = mom_of_step(I, step0 + 1);
    // the tile [ox, ox1) x [oy, oy1) and its region
    const bool wx = I.wall[0] != 0, wy = I.wall[1] != 0;
    const int ox = bx ? g.ex + bx * g.tx : 0, ox1 = bx + 1 < g.ntx ? g.ex + (bx + 1) * g.tx : I.nx;
    const int oy = by ? g.ey + by * g.ty : 0, oy1 = by + 1 < g.nty ? g.ey + (by + 1) * g.ty : I.ny;
    const int rx0 = wx ? max(ox - H, 0) : ox - H, rx1 = wx ? min(ox1 + H, I.nx) : ox1 + H;
    const int ry0 = wy ? max(oy - H, 0) : oy - H, ry1 = wy ? min(oy1 + H, I.ny) : oy1 + H;
    const int RX = rx1 - rx0, RY = ry1 - ry0;  // (at most N each; origins even)

    // this thread's cells: columns 2 l + q, rows 4 w + r.  Bit 2 r + q of in,
    // own: in the region, in the tile; pub: neighbouring regions hold it.  off:
    // byte offset of a row's pair in a plane (x even: a pair is one aligned
    // 8-byte access; where only the first cell is in the region, the second is
    // in the row's padding).  flip: bit r set where row r lies an odd number of
    // odd periods away, so that its colours are the other ones
    // (the masks are bytes of one word, the offsets wait in shared memory:
    // registers are what the sweeps are short of)
    constexpr unsigned IN = 0, OWN = 8, PUB = 16, FLIP = 24;
    unsigned off[4], mask = 0;
    {
        unsigned in = 0, own = 0, pub = 0, flip = 0;
        int refl = 0, side;
        const int x = rx0 + 2 * l;
        unsigned cin = 0, cown = 0, cpub = 0;
        const int X = x < rx1 ? map_axis(x, I.nx, I.wall[0], 1, refl, side) : 0;
#pragma unroll
        for (int q = 0; q < 2; q++) {
            cin |= (x + q < rx1) << q;
            cown |= (x + q >= ox && x + q < ox1) << q;
            cpub |= (x + q < ox + H || x + q >= ox1 - H) << q;
        }
#pragma unroll
        for (int r = 0; r < 4; r++) {
            const int y = ry0 + 4 * w + r;
            const bool here = y < ry1;
            const int Y = here ? map_axis(y, I.ny, I.wall[1], 2, refl, side) : 0;
            in |= (here ? cin : 0u) << (2 * r);
            own |= (y >= oy && y < oy1 ? cown : 0u) << (2 * r);
            pub |= (y < oy + H || y >= oy1 - H ? 3u : cpub) << (2 * r);
            flip |= (here ? (unsigned)((Y ^ y) & 1) : 0u) << r;
            off[r] = 4u * (unsigned)(Y * I.pitch + X);
        }
        mask = in | own << OWN | (pub & own) << PUB | flip << FLIP;
        offs[tid] = make_uint4(off[0], off[1], off[2], off[3]);
    }
    auto has = [&](unsigned which, int r, int q) { return (mask >> (which + 2 * r + q)) & 1; };
    auto slot = [&](int r, int q) { return ((4 * w + r) * 2 + q) * 32 + l; };
    auto load2 = [&](float *p, int r) {
        float2 v = make_float2(0.f, 0.f);
        if (has(IN, r, 0)) v = *(const float2 *)((const char *)p + off[r]);
        if (!has(IN, r, 1)) v.y = 0.f;
        return v;
    };

    // 1. colour fractions (phi_R, phi_B) of the region and the ring around it:
    //    rows -1, RY with columns -1 .. RX, then columns -1, RX
    auto fractions = [&](float rR, float rB) {
        const float xr = rR * I.inv_rhoR0, xb = rB * I.inv_rhoB0;
        return make_float2(fdiv(xr, xr + xb), fdiv(xb, xr + xb));
    };
    float2 rR[4], rB[4];
#pragma unroll
    for (int r = 0; r < 4; r++) {
        rR[r] = load2(m.rR, r);
        rB[r] = load2(m.rB, r);
    }
    {
        const int rows = 2 * (RX + 2), k = tid - rows;
        const bool top = tid >= RX + 2, right = k >= RY;
        const int x = k < 0 ? tid - (top ? RX + 2 : 0) - 1 : right ? RX : -1;
        const int y = k < 0 ? (top ? RY : -1) : k - (right ? RY : 0);
        if (k < 2 * RY) {
            int refl = 0, side;
            const int Xc = map_axis(rx0 + x, I.nx, I.wall[0], 1, refl, side);
            const int Yc = map_axis(ry0 + y, I.ny, I.wall[1], 2, refl, side);
            const unsigned o = 4u * (unsigned)(Yc * I.pitch + Xc);
            Fr[((y + 1) * 2 + (x & 1)) * FS + ((x + 2) >> 1)] = fractions(at(m.rR, o), at(m.rB, o));
        }
    }
    unsigned blue = 0;
#pragma unroll
    for (int r = 0; r < 4; r++) {
        blue |= (unsigned)(colour_fn(I, rR[r].x, rB[r].x) <= 0.f) << (2 * r);
        blue |= (unsigned)(colour_fn(I, rR[r].y, rB[r].y) <= 0.f) << (2 * r + 1);
        float2 *f = Fr + (4 * w + r + 1) * 2 * FS + l + 1;
        if (has(IN, r, 0)) f[0] = fractions(rR[r].x, rB[r].x);
        if (has(IN, r, 1)) f[FS] = fractions(rR[r].y, rB[r].y);
    }
    // the starting guess (left in the second buffers by the kernel before) and
    // the right-hand sides, in flight during the gradient
    float2 X[4][2], b[4][2];
#pragma unroll
    for (int r = 0; r < 4; r++) {
        const float2 p = load2(I.psi2, r), c = load2(I.C2, r);
        const float2 u = load2(I.rpsi, r), v = load2(I.rC, r);
        X[r][0] = make_float2(p.x, c.x);
        X[r][1] = make_float2(p.y, c.y);
        b[r][0] = make_float2(u.x, v.x);
        b[r][1] = make_float2(u.y, v.y);
    }
    // (chi waits in the weights' place until they are formed; behind the loads
    // above, not before them: 0.9 us less at 256 x 1024)
#pragma unroll
    for (int r = 0; r < 4; r++) {
        Ws[slot(r, 0)].y = chi_of(I, rR[r].x, rB[r].x);
        Ws[slot(r, 1)].y = chi_of(I, rR[r].y, rB[r].y);
    }
    const bool seam = __syncthreads_or(mask >> FLIP) != 0;  // (of an odd periodic y axis)
    // 2. gradient and weights of t+1 (grad2_cell_from): the tile's go to the
    //    planes that the next step and the exports read
#pragma unroll 1
    for (int r = 0; r < 4; r++) {
        if (!has(IN, r, 0)) break;
        // (f: of the row's column 2 l; the odd columns FS further)
        const float2 *f = Fr + (4 * w + r + 1) * 2 * FS + l + 1;
        float gx[2], gy[2], a[2], chi[2];
#pragma unroll
        for (int q = 0; q < 2; q++) {
            const bool bs = (blue >> (2 * r + q)) & 1;
            const float *c0 = bs ? &f[0].x : &f[0].y;
            gx[q] = gy[q] = 0.f;
#pragma unroll
            for (int i = 1; i < Q9; i++) {
                const int c = q + ex9(i);  // column 2 l + c
                const float v = c0[2 * (ey9(i) * 2 * FS + (c & 1) * FS + (c < 0 ? -1 : c >> 1))];
                gx[q] += w9<float>(i) * float(ex9(i)) * v;
                gy[q] += w9<float>(i) * float(ey9(i)) * v;
            }
            const float c = bs ? 6.f : -6.f;
            gx[q] *= c;
            gy[q] *= c;
            a[q] = sqrt(gx[q] * gx[q] + gy[q] * gy[q]);
            chi[q] = Ws[slot(r, q)].y;
            Ws[slot(r, q)] = make_float2(a[q] + I.eps_w, chi[q] + I.eps_w);
        }
        // (a tile's cells are grid cells: no mapping)
        const unsigned o = 4u * (unsigned)((ry0 + 4 * w + r) * I.pitch + rx0 + 2 * l);
        if (has(OWN, r, 1)) {
            *(float2 *)&at(I.gx, o) = make_float2(gx[0], gx[1]);
            *(float2 *)&at(I.gy, o) = make_float2(gy[0], gy[1]);
            *(float2 *)&at(I.a, o) = make_float2(a[0], a[1]);
            *(float2 *)&at(I.chi, o) = make_float2(chi[0], chi[1]);
        } else if (has(OWN, r, 0)) {
            at(I.gx, o) = gx[0];
            at(I.gy, o) = gy[0];
            at(I.a, o) = a[0];
            at(I.chi, o) = chi[0];
        }
    }
    __syncthreads();
    // 3. coefficients of the rows: faces h (w_c + w_nb) / 2 of Eq. 28 towards +x
    //    and +y (the other two are those of the neighbours; none across a wall
    //    or the region's edge), 1 / (w + their sum)
    float2 fE[4][2], fN[4][2], fW[4], fS[2], iv[4][2];
    // rows 4 w - 1 and 4 w + 4 (clamped: the region's edge rows have no
    // coefficient towards them)
    const int rowS = max(4 * w - 1, 0), rowN = min(4 * w + 4, N - 1);
    {
        const float hp = 0.25f * I.Ds, hc = 0.25f * I.Db;
        auto face = [&](bool on, float2 a, float2 n) {
            return make_float2(on ? __fmul_rn(hp, a.x + n.x) : 0.f,
                               on ? __fmul_rn(hc, a.y + n.y) : 0.f);
        };
        float2 below[2] = {Ws[rowS * 64 + l], Ws[rowS * 64 + 32 + l]};
        float2 row[2] = {Ws[slot(0, 0)], Ws[slot(0, 1)]};
#pragma unroll
        for (int q = 0; q < 2; q++) fS[q] = face(has(IN, 0, q) && w > 0, row[q], below[q]);
#pragma unroll
        for (int r = 0; r < 4; r++) {
            const int ry = 4 * w + r;
            const int up = r < 3 ? (ry + 1) * 64 : rowN * 64;
            const float2 above[2] = {Ws[up + l], Ws[up + 32 + l]};
            const float2 left = Ws[ry * 64 + 32 + max(l - 1, 0)];
            const float2 right = Ws[ry * 64 + min(l + 1, 31)];
            fW[r] = face(has(IN, r, 0) && l > 0, row[0], left);
            fE[r][0] = face(has(IN, r, 1), row[0], row[1]);
            fE[r][1] = face(has(IN, r, 1) && 2 * l + 2 < RX, row[1], right);
#pragma unroll
            for (int q = 0; q < 2; q++) {
                const bool here = has(IN, r, q);
                fN[r][q] = face(here && ry + 1 < RY, row[q], above[q]);
                const float2 w_ = q ? fE[r][0] : fW[r], s_ = r ? fN[r ? r - 1 : 0][q] : fS[q];
                const float dx = row[q].x + (((fE[r][q].x + fN[r][q].x) + w_.x) + s_.x);
                const float dy = row[q].y + (((fE[r][q].y + fN[r][q].y) + w_.y) + s_.y);
                iv[r][q] = make_float2(here ? fdiv(1.f, dx) : 0.f, here ? fdiv(1.f, dy) : 0.f);
                Bs[slot(r, q)] = b[r][q];
                row[q] = above[q];
            }
        }
    }
    __syncthreads();
    // (from here on the weights serve the total: zero outside the tile.)  This
    // warp's outer rows go to Xs, which has two copies of the rows that are
    // read across warps (rows 4 w and 4 w + 3 of the copy cp): half-sweeps read
    // one and write the other, so two cells of one colour that meet at a seam
    // both see the value before the half-sweep
    auto put = [&](int cp) {
#pragma unroll
        for (int q = 0; q < 2; q++) {
            Xs[slot(cp, q)] = X[0][q];
            Xs[slot(3 - cp, q)] = X[3][q];
        }
    };
#pragma unroll
    for (int r = 0; r < 4; r++)
#pragma unroll
        for (int q = 0; q < 2; q++)
            if (!has(OWN, r, q)) Ws[slot(r, q)] = make_float2(0.f, 0.f);
    put(0);
    put(1);
    const bool live = 4 * w < RY;  // (the warp has rows of the region)
    if (tid == 0) st.M0 = ctl->M0;
    __syncthreads();

    // 4. phases of NR rounds
    int rounds = 0;
    bool conv = false, keep = false;       // keep: the result is the kept round's
    float before = 0.f;                    // the round's largest update
    unsigned int bt = 0;
#pragma unroll 1
    for (int ph = 0;; ph++) {
        float th = 0.f, tl = 0.f, tr = 0.f;  // the thread's sum, of the last round
#pragma unroll 1
        for (int n = 0; n < NR; n++) {
            float2 md = make_float2(0.f, 0.f), mx = make_float2(0.f, 0.f);
            auto fold = [&](float2 d, float2 x, bool mine) {
                if (mine) {
                    md.x = fmaxf(md.x, fabsf(d.x));
                    md.y = fmaxf(md.y, fabsf(d.y));
                    mx.x = fmaxf(mx.x, fabsf(x.x));
                    mx.y = fmaxf(mx.y, fabsf(x.y));
                }
            };
            // (the last sweep's updates count, and it rounds them before it adds
            // them, which the others do not: sor_tile2_cb's roundings.  Two bodies:
            // one with the choice inside takes 0.3 us more at 64 x 517, 0.9 at 256
            // x 1024)
            auto sweep = [&](auto last) {
                constexpr bool LAST = decltype(last)::value;
                auto update = [&](int r, int q, float2 side, float2 xso, float2 xno) {
                    float2 x = fma2(fE[r][q], q ? side : X[r][1], Bs[slot(r, q)]);
                    x = fma2(fN[r][q], xno, x);
                    x = fma2(q ? fE[r][0] : fW[r], q ? X[r][0] : side, x);
                    x = fma2(r ? fN[r ? r - 1 : 0][q] : fS[q], xso, x);
                    const float2 o = X[r][q];
                    x = fma2(x, iv[r][q], make_float2(-o.x, -o.y));
                    if (LAST) {
                        const float2 d = make_float2(__fmul_rn(I.omega, x.x), __fmul_rn(I.omega, x.y));
                        X[r][q] = make_float2(__fadd_rn(o.x, d.x), __fadd_rn(o.y, d.y));
                        fold(d, X[r][q], has(OWN, r, q));
                    } else {
                        X[r][q] = make_float2(fmaf(I.omega, x.x, o.x), fmaf(I.omega, x.y, o.y));
                    }
                };
                // half-sweep t reads copy t of the rows at the warps' edges (row
                // 4 w - 1 is row 3 of the warp below, row 4 w + 4 row 0 of the one
                // above) and writes copy 1 - t
                if (!seam) {
#pragma unroll
                    for (int t = 0; t < 2; t++) {
                        if (live) {
                            // cells of colour t: cell q of row r, q = (t + r) & 1
                            const float2 xs = Xs[((w ? 4 * w - 1 - t : t) * 2 + t) * 32 + l];
                            const float2 xn = Xs[((w < NW - 1 ? 4 * w + 4 + t : N - 1) * 2 + 1 - t) * 32 + l];
                            float2 o[4];
#pragma unroll
                            for (int r = 0; r < 4; r++)
                                o[r] = ((t + r) & 1) ? shfl_down2(X[r][0]) : shfl_up2(X[r][1]);
#pragma unroll
                            for (int r = 0; r < 4; r++) {
                                const int q = (t + r) & 1;
                                update(r, q, o[r], r ? X[r ? r - 1 : 0][q] : xs,
                                       r < 3 ? X[r < 3 ? r + 1 : 3][q] : xn);
                            }
                            put(1 - t);
                        }
                        __syncthreads();
                    }
                } else {
                    // rows beyond the seam have the other colours: cell
                    // q = (t + r + flip) & 1 of row r (the same for the whole
                    // warp); where the row below updates the same column, its
                    // value before the half-sweep counts
#pragma unroll 1
                    for (int t = 0; t < 2; t++) {
                        if (live) {
                            float2 o[4];
#pragma unroll
                            for (int r = 0; r < 4; r++) {
                                const int q = (t + r + (mask >> (FLIP + r))) & 1;
                                const float2 v = q ? X[r][0] : X[r][1];
                                o[r] = make_float2(__shfl_sync(0xffffffffu, v.x, l + 2 * q - 1),
                                                   __shfl_sync(0xffffffffu, v.y, l + 2 * q - 1));
                            }
                            const int kS = (w ? 4 * w - 1 - t : t) * 64 + l;
                            const int kN = (w < NW - 1 ? 4 * w + 4 + t : N - 1) * 64 + l;
                            float2 old = make_float2(0.f, 0.f);
                            int qb = -1;  // column of the row below's update
#pragma unroll
                            for (int r = 0; r < 4; r++) {
                                const int q = (t + r + (mask >> (FLIP + r))) & 1;
                                float2 xso = r ? (q ? X[r ? r - 1 : 0][1] : X[r ? r - 1 : 0][0])
                                               : Xs[kS + 32 * q];
                                if (q == qb) xso = old;
                                qb = q;
                                if (q) {
                                    old = X[r][1];
                                    update(r, 1, o[r], xso, r < 3 ? X[r < 3 ? r + 1 : 3][1] : Xs[kN + 32]);
                                } else {
                                    old = X[r][0];
                                    update(r, 0, o[r], xso, r < 3 ? X[r < 3 ? r + 1 : 3][0] : Xs[kN]);
                                }
                            }
                            put(1 - t);
                        }
                        __syncthreads();
                    }
                }
            };
#pragma unroll 1
            for (int k = 0; k < K - 1; k++) sweep(std::false_type());
            sweep(std::true_type());
            // the round's maxima and the surfactant of the tile: products exact
            // as hi + lo, sums compensated
            float2 hi = make_float2(0.f, 0.f), lo = make_float2(0.f, 0.f);
#pragma unroll
            for (int r = 0; r < 4; r++)
#pragma unroll
                for (int q = 0; q < 2; q++) {
                    const float2 wt = Ws[slot(r, q)];
                    comp_add_prod(hi.x, lo.x, wt.x, X[r][q].x);
                    comp_add_prod(hi.y, lo.y, wt.y, X[r][q].y);
                    if (n + 1 < NR) Sn[slot(r, q)] = X[r][q];
                }
            th = hi.x;
            tl = lo.x;
            tr = 0.f;
            add3(th, tl, tr, hi.y, lo.y, 0.f);
            if (n + 1 < NR) {
                strip[0][tid] = th;
                strip[1][tid] = tl;
                strip[2][tid] = tr;
            }
            md.x = warp_max_pos(md.x);
            md.y = warp_max_pos(md.y);
            mx.x = warp_max_pos(mx.x);
            mx.y = warp_max_pos(mx.y);
            if (l == 0) *(float4 *)&redm[w][4 * n] = make_float4(md.x, md.y, mx.x, mx.y);
        }
        // publish the tile's cells that neighbouring regions hold
        float *po = (ph & 1) ? I.psi2 : I.psi, *co = (ph & 1) ? I.C2 : I.C;
        const uint4 o4 = offs[tid];
        const unsigned o[4] = {o4.x, o4.y, o4.z, o4.w};
#pragma unroll
        for (int r = 0; r < 4; r++) {
            if (has(PUB, r, 1)) {  // (then the first cell is the tile's too)
                *(float2 *)&at(po, o[r]) = make_float2(X[r][0].x, X[r][1].x);
                *(float2 *)&at(co, o[r]) = make_float2(X[r][0].y, X[r][1].y);
            } else if (has(PUB, r, 0)) {
                at(po, o[r]) = X[r][0].x;
                at(co, o[r]) = X[r][0].y;
            }
        }
        {
            float sh[NR], sl[NR], sr[NR];
#pragma unroll
            for (int n = 0; n < NR; n++) {
                sh[n] = n + 1 < NR ? strip[0][tid] : th;
                sl[n] = n + 1 < NR ? strip[1][tid] : tl;
                sr[n] = n + 1 < NR ? strip[2][tid] : tr;
            }
            if (live) lane_sum3<NR>(sh, sl, sr, nb < kSolveFine);  // (else zeros)
            if (l == 0)
#pragma unroll
                for (int n = 0; n < NR; n++) {
                    reds[0][n][w] = sh[n];
                    reds[1][n][w] = sl[n];
                    reds[2][n][w] = sr[n];
                }
        }
        __syncthreads();
        // the tile's record, the grid barrier (see grid_barrier), everybody's
        // records (32 a warp), the decision
        SolveRec *recs = (SolveRec *)I.part + (ph & 1) * kSolveMaxBlocks;
        bt += (unsigned)nb;
        if (w == 0) {
            // (lane k + 8 j: maximum k of warps 4 j .. 4 j + 3)
            const float *p = &redm[(l >> 3) * 4][l & 7];
            float v = fmaxf(fmaxf(p[0], p[8]), fmaxf(p[16], p[24]));
            v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 8));
            v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 16));
            float sh[NR], sl[NR], sr[NR];
#pragma unroll
            for (int n = 0; n < NR; n++) {
                sh[n] = reds[0][n][l & (NW - 1)];
                sl[n] = reds[1][n][l & (NW - 1)];
                sr[n] = reds[2][n][l & (NW - 1)];
            }
            lane_sum3<NR>(sh, sl, sr, true, NW / 2);
            auto whole = [&](int n) { return (double(sh[n]) + double(sl[n])) + double(sr[n]); };
            const double2 s = make_double2(whole(0), NR > 1 ? whole(NR - 1) : 0.0);
            if (l < 8) recs[blk].m[l] = v;
            if (l == 0) recs[blk].sum = s;
            __syncwarp();
            if (l == 0) {
                // (release: the block's writes before its last barrier, and the
                // record.  Relaxed polls: an acquire empties the L1 every time)
                int ok = barrier_arrive(ctl, bt, max_looks);
                const volatile unsigned int *count = &ctl->bar_count;
                for (long long looks = 0; ok && *count < bt;)
                    if (++looks > max_looks) ok = 0;
                if (!ok) atomicOr(&ctl->status, int(ST_TIMEOUT));
                __threadfence();
                st.ok = ok;
            }
        }
        __syncthreads();
        if (!st.ok) return;
        // the halo as the neighbours have it now (needed if another phase
        // follows; in flight during the decision)
#pragma unroll
        for (int r = 0; r < 4; r++)
            if (has(IN, r, 0) && !has(OWN, r, 0)) {
                const float2 p = __ldcg((const float2 *)&at(po, o[r]));
                const float2 c = __ldcg((const float2 *)&at(co, o[r]));
                X[r][0] = make_float2(p.x, c.x);
                if (has(IN, r, 1)) X[r][1] = make_float2(p.y, c.y);
            }
        if (32 * w < nb) {
            float4 v[NR];
#pragma unroll
            for (int n = 0; n < NR; n++)
                v[n] = tid < nb ? __ldcg((const float4 *)&recs[tid].m[4 * n])
                                : make_float4(0.f, 0.f, 0.f, 0.f);
            if (tid < nb) sums[tid] = __ldcg(&recs[tid].sum);
#pragma unroll
            for (int n = 0; n < NR; n++) {
                v[n] = make_float4(warp_max_pos(v[n].x), warp_max_pos(v[n].y), warp_max_pos(v[n].z),
                                   warp_max_pos(v[n].w));
                if (l == 0) *(float4 *)&redb[w][4 * n] = v[n];
            }
        }
        put(0);
        __syncthreads();
        // the decision, by every thread alike
        bool stop = false;
#pragma unroll
        for (int n = 0; n < NR; n++)
            if (!stop) {
                float mm[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 1
                for (int j = 0; 32 * j < nb; j++) {
                    const float4 v = *(const float4 *)&redb[j][4 * n];
                    mm[0] = fmaxf(mm[0], v.x);
                    mm[1] = fmaxf(mm[1], v.y);
                    mm[2] = fmaxf(mm[2], v.z);
                    mm[3] = fmaxf(mm[3], v.w);
                }
                conv = solve_converged(mm, before, rounds == 0, I.sor_tol);
                before = fmaxf(mm[0], mm[1]);
                keep = n + 1 < NR;
                rounds++;
                stop = conv || rounds >= max_rounds;
            }
        if (stop) break;
    }
    // 5. the round's total, and the rescale: x (1 + d), d = M0 / total - 1,
    //    rounded without bias (rescale_one)
    const float2 *res = keep ? Sn : Xs;
    __syncthreads();  // (the halo's copies in Xs have been written)
    if (!keep)
#pragma unroll
        for (int r = 0; r < 4; r++)
#pragma unroll
            for (int q = 0; q < 2; q++) Xs[slot(r, q)] = X[r][q];
    double total = 0.0, scale = 1.0;
    if (w == 0) {
        const bool second = NR > 1 && !keep;
        for (int k = l; k < nb; k += 32) total += second ? sums[k].y : sums[k].x;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
        if (l == 0) {
            if (total > 0) scale = st.M0 / total;
            st.dscale = float(scale - 1.0);
        }
    }
    __syncthreads();
    const float dscale_f = st.dscale;
#pragma unroll 1
    for (int k = 0; k < 8; k++) {
        if (!((mask >> (OWN + k)) & 1)) continue;
        const int x = rx0 + 2 * l + (k & 1), y = ry0 + 4 * w + (k >> 1);  // (of the tile: grid cells)
        const unsigned c = (unsigned)(y * I.pitch + x);
        const float2 v = res[slot(k >> 1, k & 1)];
        at(I.psi, 4u * c) = rescale_one(v.x, 0.0, dscale_f, rescale_key(c, 0, step0));
        at(I.C, 4u * c) = rescale_one(v.y, 0.0, dscale_f, rescale_key(c, 1, step0));
    }
    if (blk != 0 || tid != 0) return;
    ctl->pre = total;
    ctl->scale = scale;
    ctl->dscale = scale - 1.0;
    ctl->dscale_f = dscale_f;
    // (atomic: another block may be giving up its wait)
    if (!conv) atomicOr(&ctl->status, int(ST_NOCONV));
    if (!isfinite(total)) {
        atomicOr(&ctl->status, int(ST_DIVERGED));
        ctl->dead = 1;
    }
    ctl->sor_iters = rounds * K;
    ctl->sor_iters_parity = 0;
    ctl->sor_exec = 0;
    ctl->step += 1;
}

template <int K, int NR>
__global__ void __launch_bounds__(kSolveThreads, 1)
    k_solve2(Inst<float> I, SolveGeom g, int max_rounds, long long max_looks) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    solve2_tile<K, NR>(I, g, blockIdx.x % g.ntx, blockIdx.x / g.ntx, blockIdx.x, gridDim.x,
                       max_rounds, max_looks, smem_raw);
}

}  // namespace lbs
