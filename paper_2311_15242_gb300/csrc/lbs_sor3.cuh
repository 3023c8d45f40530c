// lbs_sor3.cuh — the red-black SOR of a 3D solve (arXiv 2311.15242, Sec. 2.2;
// FP32 arithmetic) as one cooperative launch: whole sweeps, each a single pass
// over the grid that marches through z, with a grid barrier between sweeps.
//
// A block owns a tile of columns (x, y) over a chunk of z and marches through
// the chunk's planes.  Lane l of warp w holds the cell pairs 2 l, 2 l + 1 of the
// region's rows 2 w, 2 w + 1 (the tile and a halo of two cells): psi, C and the
// weights a + eps, chi + eps of the planes k .. k + 2 in registers, plane k + 3 on
// its way from memory.  Step k updates red on plane k + 1 and black on plane k,
// so that a sweep reads every plane once; the red cells of a ring of one cell
// around the tile are updated too, by the neighbouring block's own arithmetic.
// The x-neighbour outside the pair comes by shuffle, the y-neighbours of other
// warps through shared memory (a ring of four planes: one block barrier a
// step), the z-neighbours are the thread's own registers.  With chunks that
// begin at even planes and regions at even rows, the column of a pair that a
// step updates is known at compile time.
//
// The update is that of k_sor_rb3, operation by operation, so the iterates are
// its own.  psi and C are read from one buffer and written to the other.
//
// What bounds it: the latency of a step (loads, a block barrier, two chains of six
// faces) with 16 warps an SM; a sweep reads 24 and writes 8 bytes a cell.
// k_sor_rb3 takes two launches of a graph loop a sweep, 24 bytes a cell and
// 6-point gathers from L1 each.  All sweeps of a step: 256 x 128 x 128 (7 sweeps)
// 753 -> 485 us, 75 x 75 x 150 (6) 252 -> 140, 100 cubed (7) 266 -> 160.
#pragma once

#include <type_traits>

#include "lbs_k3d.cuh"
#include "lbs_launch3.h"
#include "lbs_solve2.cuh"

namespace lbs {

constexpr int kSor3Rows = 32;  // rows of a region
constexpr int kSor3Threads = 512;
constexpr int kSor3H = 2;
constexpr size_t kSor3Smem = 2 * 4 * (size_t)kSor3Rows * 64 * sizeof(float2);

// tiles of an nx x ny x nz grid for `blocks` blocks at once, each taking tiles b,
// b + blocks, ...: as few columns of tiles as the region allows and the number of
// chunks of z with the shortest march (a chunk marches through three planes more
// than it owns)
inline bool sor3_geom(int nx, int ny, int nz, const int *wall, int blocks, Sor3Geom &g) {
    const int many = 1 << 20;
    if (!solve_axis(nx, wall[0] != 0, kSor3H, kSolveRegion, 1, many, g.ntx, g.tx, g.ex) ||
        !solve_axis(ny, wall[1] != 0, kSor3H, kSor3Rows, 1, many, g.nty, g.ty, g.ey))
        return false;
    const long long cols = (long long)g.ntx * g.nty;
    long long best = -1;
    for (int m = 1; m <= (nz + 1) / 2; m++) {
        int tz = (nz + m - 1) / m;
        tz += tz & 1;
        const int nt = (nz + tz - 1) / tz;
        const long long cost = (cols * nt + blocks - 1) / blocks * (tz + 3);
        if (best < 0 || cost < best) {
            best = cost;
            g.tz = tz;
            g.ntz = nt;
        }
    }
    return cols * g.ntz < (1ll << 30);
}

__global__ void __launch_bounds__(kSor3Threads, 1)
    k_sor_fs3(Inst<float> I, Sor3Geom g, int max_rounds, long long max_looks) {
    extern __shared__ __align__(16) unsigned char smem_raw[];
    float2 *Xs = (float2 *)smem_raw;                  // [slot][row][q][lane]
    float2 *Ws = Xs + 4 * kSor3Rows * 64;
    __shared__ __align__(16) float redm[kSor3Threads / 32][4];
    __shared__ int s_stop;
    const int tid = threadIdx.x, l = tid & 31, w = tid >> 5;
    Ctl *ctl = I.ctl;
    auto has = [](unsigned m, int r, int q) { return (m >> (2 * r + q)) & 1; };
    const long long plane = (long long)I.ny * I.pitch;
    const float hp = 0.5f * I.Ds, hc = 0.5f * I.Db;
    // plane p of the grid (its index), or -1 beyond a wall
    auto zmap = [&](int p) {
        int refl = 0, side;
        const int z = map_axis(p, I.nz, I.wall[2], 4, refl, side);
        return refl ? -1 : z;
    };
    const int tiles = g.ntx * g.nty * g.ntz;
    unsigned int bt = 0;
    int round = 0;
#pragma unroll 1
    for (;; round++) {
        const float *pin = (round & 1) ? I.psi2 : I.psi, *cin = (round & 1) ? I.C2 : I.C;
        float *pout = (round & 1) ? I.psi : I.psi2, *cout = (round & 1) ? I.C : I.C2;
        float v0 = 0.f, v1 = 0.f, v2 = 0.f, v3 = 0.f;
#pragma unroll 1
        for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
            const int bx = tile % g.ntx, by = (tile / g.ntx) % g.nty;
            const int bz = tile / (g.ntx * g.nty);
            const bool wx = I.wall[0] != 0, wy = I.wall[1] != 0;
            const int ox = bx ? g.ex + bx * g.tx : 0, ox1 = bx + 1 < g.ntx ? g.ex + (bx + 1) * g.tx : I.nx;
            const int oy = by ? g.ey + by * g.ty : 0, oy1 = by + 1 < g.nty ? g.ey + (by + 1) * g.ty : I.ny;
            const int rx0 = wx ? max(ox - kSor3H, 0) : ox - kSor3H, rx1 = wx ? min(ox1 + kSor3H, I.nx) : ox1 + kSor3H;
            const int ry0 = wy ? max(oy - kSor3H, 0) : oy - kSor3H, ry1 = wy ? min(oy1 + kSor3H, I.ny) : oy1 + kSor3H;
            const int RX = rx1 - rx0, RY = ry1 - ry0;
            const int zs = bz * g.tz, ze = min(zs + g.tz, I.nz);
            // this thread's pairs: bit 2 r + q of in, own; byte offset in a plane
            unsigned off[2], in = 0, own = 0;
            {
                int refl = 0, side;
                const int x = rx0 + 2 * l;
                const int X = x < rx1 ? map_axis(x, I.nx, I.wall[0], 1, refl, side) : 0;
#pragma unroll
                for (int r = 0; r < 2; r++) {
                    const int y = ry0 + 2 * w + r;
                    const bool here = y < ry1;
                    const int Y = here ? map_axis(y, I.ny, I.wall[1], 2, refl, side) : 0;
                    off[r] = 4u * (unsigned)(Y * I.pitch + X);
#pragma unroll
                    for (int q = 0; q < 2; q++) {
                        in |= (unsigned)(here && x + q < rx1) << (2 * r + q);
                        own |= (unsigned)(x + q >= ox && x + q < ox1 && y >= oy && y < oy1) << (2 * r + q);
                    }
                }
            }
            // a row's pair of a field on plane z (zeros outside the region or the grid;
            // the second cell of an odd row's last pair is padding, zero in psi and C
            // since the state was initialised or loaded: faces have no weight
            // towards it, but 0 times a NaN would be one)
            auto load2 = [&](const float *f, int z, int r) {
                float2 v = make_float2(0.f, 0.f);
                if (z >= 0 && has(in, r, 0)) v = *(const float2 *)((const char *)(f + z * plane) + off[r]);
                return v;
            };
            auto load2g = [&](const float *f, int z, int r) {  // (written in this launch)
                float2 v = make_float2(0.f, 0.f);
                if (z >= 0 && has(in, r, 0))
                    v = __ldcg((const float2 *)((const char *)(f + z * plane) + off[r]));
                return v;
            };
            // planes k, k + 1, k + 2 and the one on its way: [row][column]
            float2 Xa[2][2], Xb[2][2], Xc[2][2], Xn[2][2], Wa[2][2], Wb[2][2], Wc[2][2], Wn[2][2];
            float2 Xm[2], Wm[2];            // plane k - 1, the column that step k updates
            float2 Ba[2], Bb[2][2], Bn[2][2];  // right-hand sides: black of k, k + 1, k + 2
            bool zm, za, zb, zc;            // planes k - 1 .. k + 2 are in the grid
            auto fetch = [&](int z, float2 (&X)[2][2], float2 (&W)[2][2]) {
#pragma unroll
                for (int r = 0; r < 2; r++) {
                    const float2 p = load2g(pin, z, r), c = load2g(cin, z, r);
                    const float2 a = load2(I.a, z, r), x = load2(I.chi, z, r);
                    X[r][0] = make_float2(p.x, c.x);
                    X[r][1] = make_float2(p.y, c.y);
                    W[r][0] = make_float2(a.x + I.eps_w, x.x + I.eps_w);
                    W[r][1] = make_float2(a.y + I.eps_w, x.y + I.eps_w);
                }
            };
            auto fetch_rhs = [&](int z, float2 (&B)[2][2]) {
#pragma unroll
                for (int r = 0; r < 2; r++) {
                    const float2 p = load2(I.rpsi, z, r), c = load2(I.rC, z, r);
                    B[r][0] = make_float2(p.x, c.x);
                    B[r][1] = make_float2(p.y, c.y);
                }
            };
            auto at_ = [&](int p, int row, int q) { return ((p & 3) * kSor3Rows + row) * 64 + q * 32 + l; };
            auto put = [&](int p, const float2 (&X)[2][2], const float2 (&W)[2][2]) {
#pragma unroll
                for (int r = 0; r < 2; r++)
#pragma unroll
                    for (int q = 0; q < 2; q++) {
                        Xs[at_(p, 2 * w + r, q)] = X[r][q];
                        Ws[at_(p, 2 * w + r, q)] = W[r][q];
                    }
            };
            const int rowS = max(2 * w - 1, 0), rowN = min(2 * w + 2, kSor3Rows - 1);
            // cell q of both rows on plane p: X, W its plane, (xl, wl) and (xh, wh)
            // the planes below and above (column q), bl / bh whether they are in the
            // grid, b the right-hand sides; returns through X
            auto update = [&](int p, int r, int q, float2 (&X)[2][2], const float2 (&W)[2][2], float2 xl,
                              float2 wl, bool bl, float2 xh, float2 wh, bool bh, float2 b, bool count) {
                const float2 w0 = W[r][q], x0 = X[r][q];
                float dp = w0.x, dc = w0.y, op = b.x, oc = b.y;
                auto face = [&](bool on, float2 xn, float2 wn) {
                    const float fp = on ? hp * (0.5f * (w0.x + wn.x)) : 0.f;
                    const float fc = on ? hc * (0.5f * (w0.y + wn.y)) : 0.f;
                    dp += fp;
                    dc += fc;
                    op = fmaf(fp, xn.x, op);
                    oc = fmaf(fc, xn.y, oc);
                };
                const float2 po = X[r][1 - q], qo = W[r][1 - q];
                const float2 xo = q ? shfl_down2(X[r][0]) : shfl_up2(X[r][1]);
                const float2 wo = q ? shfl_down2(W[r][0]) : shfl_up2(W[r][1]);
                if (q) {
                    face(true, po, qo);
                    face(2 * l + 2 < RX, xo, wo);
                } else {
                    face(l > 0, xo, wo);
                    face(2 * l + 1 < RX, po, qo);
                }
                const int k = r ? at_(p, rowN, q) : at_(p, rowS, q);
                const float2 xy = Xs[k], wy_ = Ws[k];
                if (r) {
                    face(true, X[0][q], W[0][q]);
                    face(2 * w + 2 < RY, xy, wy_);
                } else {
                    face(w > 0, xy, wy_);
                    face(2 * w + 1 < RY, X[1][q], W[1][q]);
                }
                face(bl, xl, wl);
                face(bh, xh, wh);
                const float d1 = I.omega * (fdiv(op, dp) - x0.x), d2 = I.omega * (fdiv(oc, dc) - x0.y);
                const float2 n = make_float2(x0.x + d1, x0.y + d2);
                if (has(in, r, q)) X[r][q] = n;
                if (count && has(own, r, q)) {
                    v0 = fmaxf(v0, fabsf(d1));
                    v1 = fmaxf(v1, fabsf(d2));
                    v2 = fmaxf(v2, fabsf(n.x));
                    v3 = fmaxf(v3, fabsf(n.y));
                }
            };
            // step k (E: its parity): store plane k + 2, fetch k + 3, red on k + 1,
            // black on k, both at column q = (r + 1 + E) & 1 of row r
            auto step = [&](auto Ec, int k) {
                constexpr int E = decltype(Ec)::value;
                put(k + 2, Xc, Wc);
                const int zn = zmap(k + 3);
                if (k + 3 <= ze + 1) fetch(zn, Xn, Wn);
                if (k + 2 <= ze) fetch_rhs(zmap(k + 2), Bn);
                if (zb && k + 1 <= ze) {
#pragma unroll
                    for (int r = 0; r < 2; r++) {
                        const int q = (r + 1 + E) & 1;
                        update(k + 1, r, q, Xb, Wb, Xa[r][q], Wa[r][q], za, Xc[r][q], Wc[r][q], zc,
                               Bb[r][q], k + 1 >= zs && k + 1 < ze);
                        Xs[at_(k + 1, 2 * w + r, q)] = Xb[r][q];
                    }
                }
                __syncthreads();
                if (k >= zs && k < ze) {
#pragma unroll
                    for (int r = 0; r < 2; r++) {
                        const int q = (r + 1 + E) & 1;
                        update(k, r, q, Xa, Wa, Xm[r], Wm[r], zm, Xb[r][q], Wb[r][q], zb, Ba[r], true);
                        // (the row below reads this row's other column: in place)
                        char *p = (char *)(pout + k * plane) + off[r], *c = (char *)(cout + k * plane) + off[r];
                        if (has(own, r, 1)) {
                            *(float2 *)p = make_float2(Xa[r][0].x, Xa[r][1].x);
                            *(float2 *)c = make_float2(Xa[r][0].y, Xa[r][1].y);
                        } else if (has(own, r, 0)) {
                            *(float *)p = Xa[r][0].x;
                            *(float *)c = Xa[r][0].y;
                        }
                    }
                }
#pragma unroll
                for (int r = 0; r < 2; r++) {
                    const int q = (r + E) & 1;  // the column of step k + 1
                    Xm[r] = Xa[r][q];
                    Wm[r] = Wa[r][q];
                    Ba[r] = Bb[r][q];
#pragma unroll
                    for (int c = 0; c < 2; c++) {
                        Xa[r][c] = Xb[r][c];
                        Wa[r][c] = Wb[r][c];
                        Xb[r][c] = Xc[r][c];
                        Wb[r][c] = Wc[r][c];
                        Xc[r][c] = Xn[r][c];
                        Wc[r][c] = Wn[r][c];
                        Bb[r][c] = Bn[r][c];
                    }
                }
                zm = za;
                za = zb;
                zb = zc;
                zc = zn >= 0;
            };
            {
                const int z0 = zmap(zs - 2), z1 = zmap(zs - 1), z2 = zmap(zs);
                fetch(z0, Xa, Wa);
                fetch(z1, Xb, Wb);
                fetch(z2, Xc, Wc);
                fetch_rhs(z1, Bb);
                zm = false;
                za = z0 >= 0;
                zb = z1 >= 0;
                zc = z2 >= 0;
#pragma unroll
                for (int r = 0; r < 2; r++) {
                    Xm[r] = Wm[r] = Ba[r] = make_float2(0.f, 0.f);
#pragma unroll
                    for (int q = 0; q < 2; q++)
                        Xn[r][q] = Wn[r][q] = Bn[r][q] = make_float2(0.f, 0.f);
                }
            }
            put(zs - 1, Xb, Wb);
            __syncthreads();
#pragma unroll 1
            for (int k = zs - 2; k < ze; k += 2) {  // (zs is even)
                step(std::integral_constant<int, 0>(), k);
                step(std::integral_constant<int, 1>(), k + 1);
            }
            __syncthreads();
        }
        // the sweep's maxima, the grid barrier, the decision
        v0 = warp_max_pos(v0);
        v1 = warp_max_pos(v1);
        v2 = warp_max_pos(v2);
        v3 = warp_max_pos(v3);
        if (l == 0) *(float4 *)redm[w] = make_float4(v0, v1, v2, v3);
        __syncthreads();
        if (tid < 4) {
            float m = 0.f;
            for (int k = 0; k < kSor3Threads / 32; k++) m = fmaxf(m, redm[k][tid]);
            atomic_max_pos(&ctl->sweep[round][tid], double(m));
            __threadfence();  // (before the arrival that the next barrier makes)
        }
        if (!grid_barrier(ctl, gridDim.x, bt, max_looks)) return;
        if (tid == 0) {
            const bool conv = round_converged<float>(ctl, round, double(I.sor_tol));
            s_stop = conv || round + 1 >= max_rounds;
            if (blockIdx.x == 0 && s_stop) {
                // (atomic: another block may be giving up its wait)
                if (!conv) atomicOr(&ctl->status, int(ST_NOCONV));
                ctl->sor_exec = round + 1;
            }
        }
        __syncthreads();
        if (s_stop) return;
    }
}

}  // namespace lbs
