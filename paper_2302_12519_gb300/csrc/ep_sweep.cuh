// ep_sweep.cuh -- sweeps of the elliptic solve over the tabulated operator (ep_tables.cuh).
//
// Rows: a thread a row, 112 bytes of coefficients and 26 neighbours all in flight together, so a sweep is two rounds
// of memory latency whatever the grid's shape.  Bound by latency while the rows stay in L2 (48^3 shell, 10.5 thousand
// voxels: 2.6 us a sweep, the z-march 8.1; 128^3 shell, 199 thousand: 5.7 against 11.6), by their bytes above that.
// A colour pass of Gauss-Seidel reads its own eighth of the rows only: 6.4 us a pass on 1.10 million voxels, where
// the march forms every flux for one voxel in eight, 32 us.
// Bricks: 36 bytes of K and place a voxel (30 x 6 x 8 bricks share their lattices' faces), 16 of fields.  Bound by
// memory latency: the lists alone stream in 32 us of the 256^3 heart's 56.2 (3.41 million voxels; the march 69.9, bound
// by its instructions, 53 million against 35).  Measured against it and dropped: a z-march over K with packed columns
// and masked loads (54 us with the surface voxels as rows; its loads wait on one another), the same with a cp.async
// ring (65 us), bricks of 6 x 6 (58.7) and 8 x 12 (91), two bricks in flight a CTA (58), all loads of a brick at
// once (61).
#pragma once

#include "ep_stencil.cuh"
#include "ep_tables.cuh"

namespace gbep {

// Loads under a predicate, else the given value: no branch, so the loads of a row or a plane are all in flight
// together.  Volatile: the iterates change between launches, not within one, but b and x_{k-1} are overwritten by
// the thread that reads them.
__device__ __forceinline__ float load_if(bool on, const float *p, float other)
{
    float x = other;
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %1, 0; @p ld.global.f32 %0, [%2]; }" : "+f"(x) : "r"((unsigned)on), "l"(p));
    return x;
}
__device__ __forceinline__ double load_if(bool on, const double *p, double other)
{
    double x = other;
    asm volatile("{ .reg .pred p; setp.ne.u32 p, %1, 0; @p ld.global.f64 %0, [%2]; }" : "+d"(x) : "r"((unsigned)on), "l"(p));
    return x;
}

// c != 0 on the bits: an FP64 comparison would cost as much as the row's arithmetic on one neighbour.
__device__ __forceinline__ bool nonzero(float c) { return c != 0.f; }
__device__ __forceinline__ bool nonzero(double c) { return ((__double2hiint(c) & 0x7fffffff) | __double2loint(c)) != 0; }

constexpr int kSweepThreads = 128;
constexpr int kBrickThreads = 32 * kTileRows;

// The forms of a tabulated sweep: rows; bricks; rows and the torso's walk.
enum SweepForm { FORM_ROWS = 0, FORM_BRICKS = 1, FORM_TORSO = 2 };
template <int FORM>
constexpr int kSweepNT = FORM == FORM_BRICKS ? kBrickThreads : FORM == FORM_TORSO ? kThreads : kSweepThreads;
// Resident CTAs asked for: 6 of rows (80 registers; 8 spill), 5 in a colour pass, whose gathers take more (176^3 heart:
// 6.4 us a pass at 5, 6.9 at 6), 4 of the torso's 256 threads (144^3 box: 36 us a sweep, 40 at 3).
template <typename real, int FORM, int MODE = M_JAC>
constexpr int kSweepMinBlocks = sizeof(real) == 8 ? 2 : FORM == FORM_BRICKS ? EP_BRICK_BLOCKS : FORM == FORM_TORSO ? 4 : kGS<MODE> ? 5 : EP_SWEEP_BLOCKS;

// What a sweep works on, from the control block and the descriptor.
template <typename real>
struct SweepOp {
    real coef;         // omega / C, or tau / C
    real cheb_w;       // Chebyshev weight (1: the basic step)
    int cform;         // kRestart | kFold | kPrev0
    int cheb;          // semi-iteration active in this sweep
    int sweep, unit, colour;
    bool check;
};

// False when the solve is finished or at its cap.  Every thread reads the control block itself, one 16-byte load
// that the SM's CTAs share through L1: the flag changes within a launch only at the cap, where every warp of the
// launch leaves here on either reading.  The launch index comes from the slot of this launch's parity, which the
// launch before wrote: counting arrivals on one address instead cost 10 ns a CTA, 17 us a sweep at 1600 CTAs.
template <typename real, int MODE>
__device__ __forceinline__ bool sweep_begin(const Inst<real> &I, int phase, SweepOp<real> &o)
{
    const int parity = phase & 1;
    Ctl *ctl = I.ctl;
    const int4 c = *reinterpret_cast<const int4 *>(ctl);   // done, cycle0, unit[2]
    const int cycle0 = c.y;
    if (c.x) return false;
    o.unit = parity ? c.w : c.z;
    o.sweep = kGS<MODE> ? o.unit >> 3 : o.unit;
    o.colour = phase;
    if (o.sweep >= I.max_iter) {
        if (threadIdx.x == 0) {
            ctl->noconv = 1;
            ctl->iters = o.sweep;
            __threadfence();
            ctl->done = 1;
        }
        return false;
    }
    o.check = (o.sweep % I.check_every) == 0;
    if (MODE == M_IE) return true;
    o.coef = I.coef_jac;
    o.cform = o.cheb = 0;
    o.cheb_w = real(1);
    if (kGS<MODE>) return true;
    int kc = o.sweep;
    if (I.eform) {   // the iterate is x0 + e: sweep 0 reads x0 (e = 0), later sweeps read e
        kc = o.sweep - cycle0;
        o.cform = (kc == 0 ? kRestart : 0) | (kc == 0 && o.sweep > 0 ? kFold : 0) | (kc == 1 ? kPrev0 : 0);
    }
    if (kCheb<MODE>) {
        o.coef = I.cheb_tau_c;
        if (kc > 0) {
            o.cheb = 1;
            if (kc < kChebTable - 1 || 2.0 * I.cheb_theta * kc > 45.0) o.cheb_w = I.cheb_table[min(kc, kChebTable - 1)];
            else o.cheb_w = (real)cheb_weight(kc, I.cheb_rho, I.cheb_theta);   // a tiny interval, not at its limit yet
        }
    }
    return true;
}

// A sweep may be launched while the one before it still runs (programmatic dependent launch): what changes between
// sweeps is read after this, the tables before.  Nothing to wait for in an ordinary launch.
__device__ __forceinline__ void after_previous_launch()
{
    cudaTriggerProgrammaticLaunchCompletion();
    cudaGridDependencySynchronize();
}

// Iterate read and written by a launch of this parity (Chebyshev: the latter holds x_{k-1} until then).  A solve's
// first launch has parity 0, so the parity is the sweep's own and the buffers are known without the control block,
// but for the first sweep of a correction-form solve, which reads x0.
template <typename real, int MODE>
__device__ __forceinline__ const real *sweep_src(const Inst<real> &I, int parity, const SweepOp<real> &o)
{
    if (kGS<MODE> || (kJac<MODE> && I.eform && o.sweep == 0)) return I.x0;
    if (MODE == M_IE) return parity ? I.ie_x : I.v[(I.ctl->step & 1) ^ 1];
    return parity ? I.x1 : I.eform ? I.x2 : I.x0;
}
template <typename real, int MODE>
__device__ __forceinline__ real *sweep_dst(const Inst<real> &I, int parity)
{
    if (kGS<MODE>) return I.x0;
    if (MODE == M_IE) return !parity ? I.ie_x : I.v[(I.ctl->step & 1) ^ 1];
    return !parity ? I.x1 : I.eform ? I.x2 : I.x0;
}

// New value of voxel q from its value u, the operator's Lu, b_q, 1/Dhat and x_{k-1}; returns the residual.
template <typename real, int MODE>
__device__ __forceinline__ real sweep_out(const Inst<real> &I, const SweepOp<real> &o, real *out, int q, real u,
                                          real Lu, real b, real d, real prev)
{
    const real r = b - Lu;
    if (o.cform & kRestart) {   // first sweep of a cycle: fold e into x0, r becomes the right-hand side
        if (o.cform & kFold) I.x0[q] += u;
        I.b[q] = r;
        out[q] = o.coef * d * r;
    } else {
        const real basic = u + o.coef * d * r;
        if (kCheb<MODE> && o.cheb) {
            if (o.cform & kPrev0) prev = real(0);
            out[q] = o.cheb_w * (basic - prev) + prev;
        } else {
            out[q] = basic;
        }
    }
    return r;
}

// The 28 values of an assembled row.
template <typename real>
__device__ __forceinline__ void row_load(const Inst<real> &I, int row, real (&c)[kRowLen])
{
    using V = typename Vec4<real>::type;
    const V *R = reinterpret_cast<const V *>(I.rows) + row;
#pragma unroll
    for (int g = 0; g < kRowLen / 4; ++g) {
        const V a = R[(size_t)g * I.nrows];
        c[4 * g] = a.x; c[4 * g + 1] = a.y; c[4 * g + 2] = a.z; c[4 * g + 3] = a.w;
    }
}

// L u = sum A(q, q') (u_q' - u_q) of a row at s = &u_q.  A zero coefficient reads nothing (its neighbour may lie off
// the grid or the domain).
template <typename real>
__device__ __forceinline__ real row_apply(const Inst<real> &I, const real (&c)[kRowLen], const real *s, real u)
{
    const int plane = I.nx * I.ny;
    real nb[26];
#pragma unroll
    for (int t = 0; t < 26; ++t) {
        nb[t] = load_if(nonzero(c[t]), s + (nb_dx(t) + I.nx * nb_dy(t) + plane * nb_dz(t)), u);
    }
    real Lu0 = real(0), Lu1 = real(0);
#pragma unroll
    for (int t = 0; t < 26; t += 2) {
        Lu0 += c[t] * (nb[t] - u);
        Lu1 += c[t + 1] * (nb[t + 1] - u);
    }
    return Lu0 + Lu1;
}

template <typename real, int MODE>
__device__ __forceinline__ real sweep_row(const Inst<real> &I, const SweepOp<real> &o, const real *src, real *out,
                                          const real (&c)[kRowLen])
{
    const int q = row_index(c[27]);
    const real u = src[q], b = I.b[q];
    if constexpr (MODE == M_IE) {   // r = f - (I + a L) x; x+ = x + r / (1 + a D), which the row holds (Eq. iejac1)
        const real r = b - u - I.alpha_ie * row_apply(I, c, src + q, u);
        out[q] = u + c[26] * r;
        return r;
    } else {
        const real prev = kCheb<MODE> && o.cheb ? out[q] : real(0);
        return sweep_out<real, MODE>(I, o, out, q, u, row_apply(I, c, src + q, u), b, c[26], prev);
    }
}

struct BrickSmem {
    float u[kTile];
    float c[4][kLat];
};

// One brick, in three rounds: the tile of u into shared memory (cp.async); the flux F = K g of every vertex of the
// list; and the transposed gradient at every tissue voxel.  A voxel takes from each of its eight vertices
// +-F0 +-F1 +-F2 with the signs of the vertex's place, so a vertex leaves c0 = F0 + F1 + F2, c1 = F0 + F1 - F2,
// c2 = F0 - F1 + F2 and c3 = -F0 + F1 + F2 and an inner voxel reads eight values instead of 24.  A boundary voxel
// drops the components towards neighbours that are not tissue: it reads F0 = (c1 + c2) / 2 and so on.
// The lists make every lane work on tissue; a thread loads its next entries while it works on these.
template <int MODE>
__device__ __forceinline__ void sweep_brick(const Inst<float> &I, const SweepOp<float> &o, const float *src,
                                            float *out, const Brick &B, BrickSmem &sm, double &acc)
{
    static_assert(kBrickThreads == 32 * kTileRows, "a warp loads one row of each tile plane");
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    const int nx = I.nx, plane = I.nx * I.ny;
    {
        const int x = B.x0 - 1 + lane, y = B.y0 - 1 + wid;
        if (x >= 0 && x < nx && y >= 0 && y < I.ny) {
            const int z0 = B.z0 > 0 ? -1 : 0, z1 = B.z0 + B.planes < I.nz ? B.planes : B.planes - 1;
            const float *g = src + (x + nx * y + plane * (B.z0 + z0));
            float *d = sm.u + 32 * (wid + kTileRows * (z0 + 1)) + lane;
            for (int z = z0; z <= z1; ++z, g += plane, d += 32 * kTileRows) cp_async_n<4>(d, g);
        }
        cp_async_commit();
    }
    // K and places of the thread's next two vertices, a pair ahead
    float4 ka0, ka1;
    float2 kb0, kb1;
    unsigned loc0 = 0, loc1 = 0;
    auto vertex = [&](int t, float4 &ka, float2 &kb, unsigned &loc) {
        if (t < B.nvert) {
            ka = __ldcs(I.lists.k4 + (B.vbase + t));
            kb = __ldcs(I.lists.k2 + (B.vbase + t));
            loc = __ldcs(I.lists.vloc + (B.vbase + t));
        }
    };
    vertex(threadIdx.x, ka0, kb0, loc0);
    vertex(threadIdx.x + kBrickThreads, ka1, kb1, loc1);
    // the thread's voxels: list entries two ahead, b and x_{k-1} one ahead
    const int q0 = B.x0 + nx * B.y0 + plane * B.z0;
    float2 e0 = make_float2(0.f, 0.f), e1 = e0;
    float b0 = 0.f, p0 = 0.f;
    auto voxel = [&](int t, float2 &e) {
        if (t < B.nout) e = __ldcs(I.lists.out + (B.obase + t));
    };
    auto place = [&](const float2 &e) {
        const int at = __float_as_int(e.y);
        return q0 + (at & 31) + nx * ((at >> 5) & 15) + plane * (at >> 9);
    };
    auto own = [&](int t, const float2 &e) {
        if (t < B.nout) {
            b0 = I.b[place(e)];
            if (kCheb<MODE> && o.cheb) p0 = out[place(e)];
        }
    };
    voxel(threadIdx.x, e0);
    cp_async_wait<0>();
    __syncthreads();
    auto flux = [&](int t, const float4 &ka, const float2 &kb, unsigned loc) {
        const int lx = loc & 31, ly = (loc >> 5) & 15, lz = loc >> 9;
        const float *u = sm.u + lx + 32 * (ly + kTileRows * lz);
        const float u0 = u[0], u1 = u[1], u2 = u[32], u3 = u[33];
        const float *v = u + 32 * kTileRows;
        const float u4 = v[0], u5 = v[1], u6 = v[32], u7 = v[33];
        float gx, gy, gz;
        if (t < B.nfull) {
            // differences first: of neighbours they are all but exact, where sums would round at the iterate's own size
            gx = ((u1 - u0) + (u3 - u2)) + ((u5 - u4) + (u7 - u6));
            gy = ((u2 - u0) + (u3 - u1)) + ((u6 - u4) + (u7 - u5));
            gz = ((u4 - u0) + (u5 - u1)) + ((u6 - u2) + (u7 - u3));
        } else {
            const unsigned w = I.lists.vpair[B.pbase + t - B.nfull];
            auto pair = [&](int bit, float lo, float hi) { return (w >> bit) & 1u ? hi - lo : 0.f; };
            gx = (pair(0, u0, u1) + pair(1, u2, u3)) + (pair(2, u4, u5) + pair(3, u6, u7));
            gy = (pair(4, u0, u2) + pair(5, u1, u3)) + (pair(6, u4, u6) + pair(7, u5, u7));
            gz = (pair(8, u0, u4) + pair(9, u1, u5)) + (pair(10, u2, u6) + pair(11, u3, u7));
        }
        const float F0 = ka.x * gx + ka.w * gy + kb.x * gz;
        const float F1 = ka.w * gx + ka.y * gy + kb.y * gz;
        const float F2 = kb.x * gx + kb.y * gy + ka.z * gz;
        float *c = sm.c[0] + lx + kLatX * (ly + kLatY * lz);
        c[0] = (F0 + F1) + F2;
        c[kLat] = (F0 + F1) - F2;
        c[2 * kLat] = (F0 - F1) + F2;
        c[3 * kLat] = (F1 - F0) + F2;
    };
    for (int t = threadIdx.x; t < B.nvert; t += 2 * kBrickThreads) {
        const float4 a = ka0, e = ka1;
        const float2 b = kb0, f = kb1;
        const unsigned la = loc0, le = loc1;
        vertex(t + 2 * kBrickThreads, ka0, kb0, loc0);
        vertex(t + 3 * kBrickThreads, ka1, kb1, loc1);
        flux(t, a, b, la);
        if (t + kBrickThreads < B.nvert) flux(t + kBrickThreads, e, f, le);
    }
    own(threadIdx.x, e0);
    voxel(threadIdx.x + kBrickThreads, e1);
    __syncthreads();
    for (int t = threadIdx.x; t < B.nout; t += kBrickThreads) {
        const int at = __float_as_int(e0.y), ox = at & 31, oy = (at >> 5) & 15, oz = at >> 9, q = place(e0);
        const float bt = b0, dt = e0.x, pt = p0;
        e0 = e1;
        own(t + kBrickThreads, e0);
        voxel(t + 2 * kBrickThreads, e1);
        const int l = ox + kLatX * (oy + kLatY * oz);
        constexpr int Y = kLatX, Z = kLatX * kLatY;
        float Lu;
        if (t < B.ninner) {
            const float *c0 = sm.c[0] + l, *c1 = sm.c[1] + l, *c2 = sm.c[2] + l, *c3 = sm.c[3] + l;
            Lu = ((c0[0] - c0[1 + Y + Z]) + (c1[Z] - c1[1 + Y])) + ((c2[Y] - c2[1 + Z]) + (c3[1] - c3[Y + Z]));
        } else {
            const unsigned f = I.lists.oflag[B.fbase + t - B.ninner];
            float x0 = 0.f, x1 = 0.f, y0 = 0.f, y1 = 0.f, z0 = 0.f, z1 = 0.f;   // twice the sums over each face
#pragma unroll
            for (int v = 0; v < 8; ++v) {
                const int m = l + (v & 1) + Y * ((v >> 1) & 1) + Z * (v >> 2);
                const float c1 = sm.c[1][m], c2 = sm.c[2][m], c3 = sm.c[3][m];
                (v & 1 ? x1 : x0) += c1 + c2;
                (v & 2 ? y1 : y0) += c1 + c3;
                (v & 4 ? z1 : z0) += c2 + c3;
            }
            auto face = [&](int bit, float s) { return (f >> bit) & 1u ? s : 0.f; };
            Lu = 0.5f * (((face(0, x0) - face(1, x1)) + (face(2, y0) - face(3, y1))) + (face(4, z0) - face(5, z1)));
        }
        const float u = sm.u[ox + 1 + 32 * (oy + 1 + kTileRows * (oz + 1))];
        const float r = sweep_out<float, MODE>(I, o, out, q, u, Lu, bt, dt, pt);
        if (o.check) acc += (double)(r * r);
    }
}

// One work item of the walk through the torso of a torso handle.  A voxel with nothing but torso around it (or the
// grid's border) sees the isotropic operator sig_o I, which needs no record: F_a = C r_a^2 nT sig_o g_a with counts
// that are constants of a lane, as in the walk over clear items (whose staging this shares: warp w copies voxel row w,
// warp 0 also the ninth).  Every voxel of the grid is walked through; those that are not of this kind are not written
// (walk_dinv < 0) and their values reach only vertices that no written voxel has.  With the rows beside it 36 us a sweep
// of the 144^3 box (2.3 million voxels walked, 0.7 million rows); the two-term items and their single-term far ones 76.
struct WalkSmem {
    static constexpr int D = 4;
    float u[D][kWarps + 1][32];
    float b[D][kWarps][32], d[D][kWarps][32], p[D][kWarps][32];
    float F[2][3][kWarps][32];
};

template <int MODE>
__device__ __forceinline__ void sweep_walk(const Inst<float> &I, const SweepOp<float> &o, const float *src, float *out,
                                           const Seg &sg, WalkSmem &sm, double &total)
{
    constexpr int D = WalkSmem::D;
    const int lane = threadIdx.x & 31, row = threadIdx.x >> 5;
    const int nx = I.nx, plane = I.nx * I.ny, nz = I.nz;
    const int x = sg.x0 - 1 + lane, y = sg.by * kTileY + row - 1;
    const bool own = x >= 0 && x < nx, left = x >= 1 && x - 1 < nx;
    const bool yl = y >= 0 && y < I.ny, yh = y + 1 < I.ny;
    const bool lo = own && yl, ninth = row == 0 && own && y + kWarps < I.ny;
    const int q0 = x + nx * y, q8 = q0 + nx * kWarps;
    const int cols = (left ? 1 : 0) + (own ? 1 : 0), rows = (yl ? 1 : 0) + (yh ? 1 : 0);
    const float ax = rcp_count<float>((float)(cols == 2 ? rows : 0)), ay = rcp_count<float>((float)(rows == 2 ? cols : 0)),
                az = rcp_count<float>((float)(cols * rows)), iso = I.C * I.sig_o * (float)(cols * rows);
    const float kx = ax * ax * iso, ky = ay * ay * iso, kz = az * az * iso;   // one plane (kz: of two, half its voxels)
    const int kbeg = sg.k0 - 1, kend = sg.k1;
    auto issue = [&](int k, int slot) {
        if (k <= kend) {
            if ((unsigned)k < (unsigned)nz) {
                if (lo) {
                    const int q = q0 + k * plane;
                    cp_async_n<4>(&sm.u[slot][row][lane], src + q);
                    if (row > 0) {
                        cp_async_n<4>(&sm.b[slot][row][lane], I.b + q);
                        cp_async_n<4>(&sm.d[slot][row][lane], I.walk_dinv + q);
                        if (kCheb<MODE> && o.cheb) cp_async_n<4>(&sm.p[slot][row][lane], out + q);
                    }
                }
                if (ninth) cp_async_n<4>(&sm.u[slot][kWarps][lane], src + (q8 + k * plane));
            } else {
                sm.u[slot][row][lane] = 0.f;
                if (row == 0) sm.u[slot][kWarps][lane] = 0.f;
            }
        }
        cp_async_commit();
    };
#pragma unroll
    for (int j = 0; j < D; ++j) {   // what no copy ever fills
        if (!lo) sm.u[j][row][lane] = 0.f;
        if (row == 0 && !ninth) sm.u[j][kWarps][lane] = 0.f;
    }
#pragma unroll
    for (int j = 0; j < D - 1; ++j) issue(kbeg + j, j);
    cp_async_wait<D - 2>();
    __syncthreads();
    const bool writes = row > 0 && lane >= 1 && lane <= kTileX && lo;
    float X = 0.f, Y = 0.f, S = 0.f, u = 0.f, h = 0.f, b = 0.f, d = -1.f, pv = 0.f, acc = 0.f;
    auto step = [&](int k, int slot) {
        const int par = k & 1;
        const float vl = sm.u[slot][row][lane], vh = sm.u[slot][row + 1][lane];
        const float bn = sm.b[slot][row][lane], dn = sm.d[slot][row][lane];
        const float pn = kCheb<MODE> ? sm.p[slot][row][lane] : 0.f;
        // differences first: of neighbours they are all but exact, where sums would round at the iterate's own size
        // (the 144^3 box took 5 to 9 % more sweeps to a residual of 1e-6 over sums)
        const float ll = __shfl_up_sync(kFull, vl, 1), lh = __shfl_up_sync(kFull, vh, 1);
        const float c = (vl - u) + (vh - h), cl = __shfl_up_sync(kFull, c, 1);
        const float Xn = (vl - ll) + (vh - lh), Yn = (vh - vl) + (lh - ll);
        float F0 = 0.f, F1 = 0.f, F2 = 0.f;
        if (k > kbeg) {   // two planes: the squared counts' 1/4 times twice the voxels
            const bool both = k > 0 && k < nz;
            const float f = both ? 0.5f : 1.f;
            F0 = kx * f * (X + Xn);
            F1 = ky * f * (Y + Yn);
            F2 = both ? 2.f * kz * (c + cl) : 0.f;
        }
        X = Xn; Y = Yn;
        sm.F[par][0][row][lane] = F0;
        sm.F[par][1][row][lane] = F1;
        sm.F[par][2][row][lane] = F2;
        issue(k + D - 1, (slot + D - 1) % D);   // the slot of plane k - 1, which every warp has read
        cp_async_wait<D - 2>();
        __syncthreads();
        const int below = row >= 1 ? row - 1 : 0;
        const float p = sm.F[par][0][below][lane] + F0, q = sm.F[par][1][below][lane] - F1, r = sm.F[par][2][below][lane] + F2;
        const float w = (p + q) + __shfl_down_sync(kFull, q - p, 1), z = r + __shfl_down_sync(kFull, r, 1);
        if (k > kbeg + 1 && writes && d >= 0.f) {
            const float res = sweep_out<float, MODE>(I, o, out, q0 + (k - 1) * plane, u, S + (w - z), b, d, pv);
            acc += res * res;
        }
        S = w + z;
        u = vl; h = vh; b = bn; d = dn; pv = pn;
    };
    for (int k = kbeg;;) {
        step(k, 0);
        if (++k > kend) break;
        step(k, 1);
        if (++k > kend) break;
        step(k, 2);
        if (++k > kend) break;
        step(k, 3);
        if (++k > kend) break;
    }
    cp_async_wait<0>();
    total += (double)acc;   // at most 32 planes in FP32, FP64 above
}

// The work of CTA `cta` of the I.nsweep CTAs of a sweep, a brick, an item of the torso's walk
// or a share of the rows, after the handle's form.
template <typename real, int MODE, int FORM>
__device__ __forceinline__ void sweep_cta(const Inst<real> &I, int phase, int cta, unsigned char *smem, double *sred,
                                          int *sflag)
{
    constexpr int NT = kSweepNT<FORM>;
    const int parity = phase & 1;
    SweepOp<real> o;
    double acc = 0.0;
    const int nwalk = FORM == FORM_TORSO ? I.nwalk : 0;
    if (FORM == FORM_TORSO && cta < nwalk) {
        if constexpr (FORM == FORM_TORSO) {
            const Seg sg = I.walk[cta];
            after_previous_launch();
            if (!sweep_begin<real, MODE>(I, phase, o)) return;
            sweep_walk<MODE>(I, o, sweep_src<real, MODE>(I, parity, o), sweep_dst<real, MODE>(I, parity), sg,
                             *reinterpret_cast<WalkSmem *>(smem), acc);
        }
    } else if constexpr (FORM == FORM_BRICKS) {
        const Brick B = I.bricks[cta];
        after_previous_launch();
        if (!sweep_begin<real, MODE>(I, phase, o)) return;
        sweep_brick<MODE>(I, o, sweep_src<real, MODE>(I, parity, o), sweep_dst<real, MODE>(I, parity), B,
                          *reinterpret_cast<BrickSmem *>(smem), acc);
    } else {
        const int r0 = kGS<MODE> ? I.row_colour[phase] : 0, r1 = kGS<MODE> ? I.row_colour[phase + 1] : I.nrows;
        int i = r0 + (cta - nwalk) * NT + threadIdx.x;
        real c[kRowLen];
        if (i < r1) row_load(I, i, c);   // constants: read while the sweep before this one ends
        after_previous_launch();
        if (!sweep_begin<real, MODE>(I, phase, o)) return;
        const real *src = sweep_src<real, MODE>(I, parity, o);
        real *out = sweep_dst<real, MODE>(I, parity);
        while (i < r1) {
            const real r = sweep_row<real, MODE>(I, o, src, out, c);
            if (o.check) {
                const float f = (float)r;
                acc += (double)(f * f);
            }
            i += (I.nsweep - nwalk) * NT;
            if (i < r1) row_load(I, i, c);
        }
    }
    if (cta == 0 && threadIdx.x == 0) I.ctl->unit[parity ^ 1] = o.unit + 1;
    if (!o.check) return;
    // FP64 partial norms, summed in a fixed order by the CTA that arrives last.  CTAs count in groups, each counter
    // on its own line, and the last of a group counts the group.
    const int part = kGS<MODE> ? o.colour : 0, parts = kGS<MODE> ? 8 : 1;
    const double tot = block_sum<NT>(acc, sred);
    if (threadIdx.x == 0) {
        I.partials[part * I.nsweep + cta] = tot;
        __threadfence();
        const int g = cta % kArriveGroups, groups = min(I.nsweep, kArriveGroups);
        const unsigned size = (unsigned)((I.nsweep - g + kArriveGroups - 1) / kArriveGroups);
        unsigned *mine = I.sweep_arrive + (g + 1) * kArriveStride;
        bool last = atomicAdd(mine, 1u) == size - 1u;
        if (last) {
            *mine = 0u;
            __threadfence();
            last = atomicAdd(I.sweep_arrive, 1u) == (unsigned)groups - 1u;
            if (last) *I.sweep_arrive = 0u;
        }
        *sflag = last && part == parts - 1;
    }
    __syncthreads();
    if (*sflag) {
        __threadfence();
        double s = 0;
        for (int i = threadIdx.x; i < parts * I.nsweep; i += NT) s += ((volatile double *)I.partials)[i];
        s = block_sum<NT>(s, sred);
        if (threadIdx.x == 0) sweep_decide(I, o.sweep, kJac<MODE> && !kGS<MODE> && I.eform, s);
    }
}

// Bytes of dynamic shared memory of a sweep CTA.
template <int FORM>
constexpr size_t kSweepSmem = FORM == FORM_BRICKS ? sizeof(BrickSmem) : FORM == FORM_TORSO ? sizeof(WalkSmem) : 0;

// Single instance.
template <typename real, int MODE, int FORM>
__global__ void __launch_bounds__(kSweepNT<FORM>, kSweepMinBlocks<real, FORM, MODE>) k_sweep(Inst<real> I, int phase)
{
    extern __shared__ __align__(16) unsigned char ep_sweep_smem[];
    __shared__ double sred[kSweepNT<FORM> / 32];
    __shared__ int sflag;
    sweep_cta<real, MODE, FORM>(I, phase, blockIdx.x, ep_sweep_smem, sred, &sflag);
}

// Batched: the sweep CTAs of all members of a list with this form (the batch's trial sweeps).
template <typename real, int MODE, int FORM>
__global__ void __launch_bounds__(kSweepNT<FORM>, kSweepMinBlocks<real, FORM>)
k_sweep_batch(const Inst<real> *insts, const BItem *items, int phase)
{
    extern __shared__ __align__(16) unsigned char ep_sweep_smem[];
    __shared__ double sred[kSweepNT<FORM> / 32];
    __shared__ int sflag;
    __shared__ Inst<real> sI;
    const BItem it = items[blockIdx.x];
    const Inst<real> &I = stage_inst(insts + it.inst, sI);
    if ((I.nbricks > 0) != (FORM == FORM_BRICKS)) return;
    sweep_cta<real, MODE, FORM>(I, phase, it.item, ep_sweep_smem, sred, &sflag);
}

// Batched: the unfinished members of a list (see k_stencil_active).  The descriptor is copied before the finished
// flag is read, so a warp that leaves early has done its share.  A CTA does `share` sweep CTAs of its member one after
// another: the lookup and the descriptor cost as much as a sweep CTA of rows itself (200 blocks of 24^3, 1 000 Jacobi
// sweeps: 86 ms with one, 80 with three).
template <typename real, int MODE, int FORM>
__global__ void __launch_bounds__(kSweepNT<FORM>, kSweepMinBlocks<real, FORM>)
k_sweep_active(const Inst<real> *insts, const ActRec *act, int n, int share, int phase)
{
    extern __shared__ __align__(16) unsigned char ep_sweep_smem[];
    __shared__ double sred[kSweepNT<FORM> / 32];
    __shared__ int sflag, sk;
    __shared__ Inst<real> sI;
    const int i = blockIdx.x;
    if (threadIdx.x == 0) sk = -1;
    __syncthreads();
    for (int k = threadIdx.x; k < n; k += blockDim.x) {
        const ActRec a = act[k];
        if (a.inst >= 0 && a.cum <= i && i < act[k + 1].cum) sk = k;
    }
    __syncthreads();
    if (sk < 0) return;
    const ActRec r = act[sk];
    const Inst<real> &I = stage_inst(insts + r.inst, sI);
    const int first = (i - r.cum) * share, last = min(first + share, I.nsweep);
    for (int cta = first; cta < last; ++cta) {
        if (cta > first) __syncthreads();   // the shared memory is used again
        sweep_cta<real, MODE, FORM>(I, phase, cta, ep_sweep_smem, sred, &sflag);
    }
}

// Explicit monodomain steps over the rows.  A step is one launch: the diffusion of v* (the new v, activation times, the
// non-finite flag), then the reaction of the next step at the same voxel (its v*, into the other of two buffers, and
// its w, into the buffer of the w that this step used up); the first step of a call is led by the reaction alone.
// The fused walk recomputes the reaction of its halo and rebuilds the tensors; in FP64, where this GPU does two
// operations a clock and SM, that is most of its time: 121 us a step of the 32^3 slab against 8.5 here.  In FP32 small
// grids are bound by latency: 61 x 45 x 53, 19.5 us a step in the walk, 7.1 with reaction and diffusion as two
// launches, 5.2 here.  Launches of step parity p read the step from tick[p] and leave tick[p ^ 1].
template <typename real>
__device__ __forceinline__ real *vstar(const Inst<real> &I, int parity)
{
    return parity ? I.x1 : I.b;   // scratch between steps
}

template <typename real>
__device__ __forceinline__ void react_voxels(const Inst<real> &I, long long step, real *vs_out, int first, int end, int stride)
{
    const int parity = (int)(step & 1);
    const double tn = (double)step * I.dt_d;
    const real *v = I.v[parity], *w = I.w[parity];
    real *wn = I.w[parity ^ 1];
    const unsigned stim = active_stimuli(I, tn);
    for (int i = first; i < end; i += stride) {
        const int q = I.idx[i];
        int x = 0, y = 0, z = 0;   // used by active stimuli only
        if (stim) {
            x = q % I.nx;
            y = (q / I.nx) % I.ny;
            z = q / (I.nx * I.ny);
        }
        real vs, ws;
        ms_step(I, stim, v[q], w[q], x, y, z, vs, ws);
        vs_out[q] = vs;
        wn[q] = ws;
    }
}

template <typename real>
__device__ __forceinline__ long long diffuse_react_rows(const Inst<real> &I, const long long *counter, const real *vs_in,
                                                        real *vs_out, int first, int end, int stride)
{
    real c[kRowLen];
    if (first < end) row_load(I, first, c);
    after_previous_launch();
    const long long step = *counter;
    const int parity = (int)(step & 1);
    const double tn = (double)step * I.dt_d;
    const real *v = I.v[parity];
    real *vn = I.v[parity ^ 1];
    const unsigned stim = active_stimuli(I, (double)(step + 1) * I.dt_d);
    for (int i = first; i < end; i += stride) {
        if (i != first) row_load(I, i, c);
        const int q = row_index(c[27]);
        const real u = vs_in[q], vold = v[q], w = I.w[parity ^ 1][q];
        const real vnew = u - I.coef_par * row_apply(I, c, vs_in + q, u);
        vn[q] = vnew;
        if (vold < real(0.5) && vnew >= real(0.5) && I.tact[q] < real(0))
            I.tact[q] = (real)(tn + I.dt_d * (0.5 - (double)vold) / ((double)vnew - (double)vold));
        if (!isfinite(vnew)) atomicOr(&I.ctl->nonfinite, 1);
        real vs, ws;
        ms_step(I, stim, vnew, w, q % I.nx, (q / I.nx) % I.ny, q / (I.nx * I.ny), vs, ws);
        vs_out[q] = vs;
        I.w[parity][q] = ws;
    }
    return step;
}

template <typename real>
__global__ void __launch_bounds__(kSweepThreads) k_react(Inst<real> I, int parity)
{
    after_previous_launch();
    react_voxels(I, I.ctl->tick[parity], vstar(I, parity), blockIdx.x * kSweepThreads + threadIdx.x, I.nrows,
                 gridDim.x * kSweepThreads);
}

template <typename real>
__global__ void __launch_bounds__(kSweepThreads, sizeof(real) == 8 ? 2 : EP_SWEEP_BLOCKS) k_mono_step(Inst<real> I, int parity)
{
    const long long step = diffuse_react_rows(I, &I.ctl->tick[parity], vstar(I, parity), vstar(I, parity ^ 1),
                                              blockIdx.x * kSweepThreads + threadIdx.x, I.nrows,
                                              gridDim.x * kSweepThreads);
    if (blockIdx.x == 0 && threadIdx.x == 0) I.ctl->tick[parity ^ 1] = step + 1;
}

// Batched: the same two launches over the members with rows; blockIdx.x an entry of the packed reduction-chunk list
// (2 048 rows), blockIdx.y a share of it, as many shares as give the GPU three rounds of resident CTAs (mono_shares):
// bound by latency, a small batch needs all its rows in flight, while in a large one each CTA's copy of the descriptor
// counts.  The reaction alone leads the launches of a call (STEP false); the step counter moves at the end of the
// batched step.  us a step in the march over recomputed tensors, in reaction and diffusion as two launches of whole
// chunks, and here: 64 slabs of 24^3 54, 65, 46; four of 24^3 33, 32, 12; four of 88^3 96, 100, 88; sixteen of 88^3
// 338, 320, 295; 32 shells of 128^3 432, 274, 240.
template <typename real, bool STEP>
__global__ void __launch_bounds__(kSweepThreads, EP_SWEEP_BLOCKS) k_mono_batch(const Inst<real> *insts, const BItem *items)
{
    __shared__ Inst<real> sI;
    const BItem it = items[blockIdx.x];
    const Inst<real> &I = stage_inst(insts + it.inst, sI);
    if (!I.tab) return;
    const long long part = (long long)it.item * gridDim.y + blockIdx.y, parts = (long long)it.nitems * gridDim.y;
    const int r0 = (int)(I.nrows * part / parts), r1 = (int)(I.nrows * (part + 1) / parts);
    const int parity = (int)(I.ctl->step & 1);
    if (STEP) diffuse_react_rows(I, &I.ctl->step, vstar(I, parity), vstar(I, parity ^ 1), r0 + threadIdx.x, r1, kSweepThreads);
    else react_voxels(I, I.ctl->step, vstar(I, parity), r0 + threadIdx.x, r1, kSweepThreads);
}

// cheb_weight(k) for k < kChebTable - 1; the last entry is the weights' limit 2 e^-theta / rho.
template <typename real>
__global__ void k_cheb_table(double rho, double theta, real *t)
{
    for (int k = threadIdx.x; k < kChebTable; k += blockDim.x)
        t[k] = (real)(k < kChebTable - 1 ? cheb_weight(k, rho, theta) : (2.0 / rho) * exp(-theta));
}

}  // namespace gbep
