// ep_tables.cuh -- the diffusion operator tabulated once at set-up, for the kernels that apply it many times.
//
// The operator is L = G'^T S G' (masked vertex gradients, vertex tensors, transposed gradient).  At a vertex the flux
// is F = K g with one symmetric 3x3 matrix K_ab = C r_a r_b (nT sT I + dS sum f f^T)_ab and g the sums of the valid
// pair differences.  Two forms:
//   rows:   for a list of voxels, the 26 coefficients A(q, q') of the assembled row (without the diagonal: rows sum
//           to zero, so L u = sum A(q, q') (u_q' - u_q)), 1/Dhat and the voxel's index, 28 values a row in seven
//           groups of four, each group contiguous over the rows;
//   bricks: blocks of 30 x kBrickY x kBrickZ voxels with the list of their vertices (K, position, and the valid
//           pairs of the vertices whose block is not all tissue) and of their tissue voxels (position, 1/Dhat, and
//           the tissue flags of the six neighbours of those that touch the tissue's surface).
// All entries are formed in FP64 from the fp32 records and rounded once.
#pragma once

#include "ep_aux.cuh"

namespace gbep {

constexpr int kRowLen = 28;       // 26 coefficients, 1/Dhat, the voxel index
// Brick of voxels, its vertex lattice (31 wide, so that the entries of a dense list are neighbours in shared memory)
// and its tile (the voxels and one layer around them, 32 wide).
constexpr int kBrickX = 30, kBrickY = EP_BRICK_Y, kBrickZ = EP_BRICK_Z;
constexpr int kLatX = kBrickX + 1, kLatY = kBrickY + 1, kLat = kLatX * kLatY * (kBrickZ + 1);
constexpr int kTileRows = kBrickY + 2, kTile = 32 * kTileRows * (kBrickZ + 2);
static_assert(kBrickY < 16 && kBrickZ < 16, "positions are packed in 5 + 4 + 4 bits");

template <typename real>
struct Vec4;
template <>
struct Vec4<float> { using type = float4; };
template <>
struct Vec4<double> { using type = double4_32a; };

// Offset t (0..25) of a row's neighbours: all (dx, dy, dz) in {-1, 0, 1}^3 but the centre, x fastest.
__host__ __device__ constexpr int nb_cell(int t) { return t < 13 ? t : t + 1; }
__host__ __device__ constexpr int nb_dx(int t) { return nb_cell(t) % 3 - 1; }
__host__ __device__ constexpr int nb_dy(int t) { return nb_cell(t) / 3 % 3 - 1; }
__host__ __device__ constexpr int nb_dz(int t) { return nb_cell(t) / 9 - 1; }

// Index bits of a row in its last value.
__device__ __forceinline__ float row_tag(int q, float) { return __int_as_float(q); }
__device__ __forceinline__ double row_tag(int q, double) { return __hiloint2double(0, q); }
__device__ __forceinline__ int row_index(float t) { return __float_as_int(t); }
__device__ __forceinline__ int row_index(double t) { return __double2loint(t); }

// Assembled rows of the operator with sigma_T = sT, sigma_L - sigma_T = dS (times C), and with so > 0 the torso
// term (records with torso voxels); one thread a row.
template <typename real>
__global__ void k_build_rows(int nx, int ny, int nz, double sT, double dS, double so, double C, const float4 *rec,
                             const int *rowq, long long nrows, const real *ie_inv, real *rows)
{
    for (long long r = blockIdx.x * (long long)blockDim.x + threadIdx.x; r < nrows;
         r += (long long)gridDim.x * blockDim.x) {
        const int q = rowq[r];
        const int i = q % nx, j = (q / nx) % ny, k = q / (nx * ny);
        double a[27];
        for (int t = 0; t < 27; ++t) a[t] = 0.0;
        for (int v = 0; v < 8; ++v) {
            const int s = v & 1, t = (v >> 1) & 1, u = v >> 2;
            int cnt[3], cntd[3], nT, nB;
            double M[6];
            bool T[2][2][2], Td[2][2][2];
            vertex_static(nx, ny, nz, rec, i + s, j + t, k + u, cnt, nT, M, T, cntd, nB, Td);
            const int os = 1 - s, ot = 1 - t, ou = 1 - u;   // q's place in the vertex's block
            if (T[ou][ot][os]) {
                const double r0 = cnt[0] ? 1.0 / cnt[0] : 0.0, r1 = cnt[1] ? 1.0 / cnt[1] : 0.0,
                             r2 = cnt[2] ? 1.0 / cnt[2] : 0.0;
                const double c0 = T[ou][ot][1 - os] ? (os ? r0 : -r0) : 0.0;
                const double c1 = T[ou][1 - ot][os] ? (ot ? r1 : -r1) : 0.0;
                const double c2 = T[1 - ou][ot][os] ? (ou ? r2 : -r2) : 0.0;
                const double iso = sT * nT;
                const double w0 = c0 * (iso + dS * M[0]) + c1 * dS * M[3] + c2 * dS * M[4];
                const double w1 = c0 * dS * M[3] + c1 * (iso + dS * M[1]) + c2 * dS * M[5];
                const double w2 = c0 * dS * M[4] + c1 * dS * M[5] + c2 * (iso + dS * M[2]);
                for (int p = 0; p < 8; ++p) {
                    const int ps = p & 1, pt = (p >> 1) & 1, pu = p >> 2;
                    if (!T[pu][pt][ps]) continue;
                    double d = 0.0;
                    if (T[pu][pt][1 - ps]) d += w0 * (ps ? r0 : -r0);
                    if (T[pu][1 - pt][ps]) d += w1 * (pt ? r1 : -r1);
                    if (T[1 - pu][pt][ps]) d += w2 * (pu ? r2 : -r2);
                    a[(s + ps) + 3 * (t + pt) + 9 * (u + pu)] += d;
                }
            }
            if (so > 0.0 && nB > 0) {
                const double r0 = cntd[0] ? 1.0 / cntd[0] : 0.0, r1 = cntd[1] ? 1.0 / cntd[1] : 0.0,
                             r2 = cntd[2] ? 1.0 / cntd[2] : 0.0;
                const double ko = so * nB;
                const double w0 = Td[ou][ot][1 - os] ? (os ? r0 : -r0) * ko : 0.0;
                const double w1 = Td[ou][1 - ot][os] ? (ot ? r1 : -r1) * ko : 0.0;
                const double w2 = Td[1 - ou][ot][os] ? (ou ? r2 : -r2) * ko : 0.0;
                for (int p = 0; p < 8; ++p) {
                    const int ps = p & 1, pt = (p >> 1) & 1, pu = p >> 2;
                    if (!Td[pu][pt][ps]) continue;
                    double d = 0.0;
                    if (Td[pu][pt][1 - ps]) d += w0 * (ps ? r0 : -r0);
                    if (Td[pu][1 - pt][ps]) d += w1 * (pt ? r1 : -r1);
                    if (Td[1 - pu][pt][ps]) d += w2 * (pu ? r2 : -r2);
                    a[(s + ps) + 3 * (t + pt) + 9 * (u + pu)] += d;
                }
            }
        }
        auto put = [&](int e, real x) { rows[((long long)(e / 4) * nrows + r) * 4 + e % 4] = x; };
        for (int t = 0; t < 26; ++t) put(t, (real)(C * a[nb_cell(t)]));
        put(26, ie_inv ? ie_inv[q] : (real)rec[q].w);   // implicit diffusion: 1 / (1 + a D)
        put(27, row_tag(q, real(0)));
    }
}

// 1/Dhat of the voxels of a torso handle that the walk takes, -1 elsewhere.
template <typename real>
__global__ void k_build_walk(long long n, const uint8_t *walked, const float4 *rec, real *dinv)
{
    for (long long q = blockIdx.x * (long long)blockDim.x + threadIdx.x; q < n; q += (long long)gridDim.x * blockDim.x)
        dinv[q] = walked[q] ? (real)rec[q].w : real(-1);
}

// Lists of every brick, one CTA a brick: vertices in lattice order, the full ones (eight tissue voxels) first, then
// the others that touch tissue; tissue voxels in window order, the inner ones (eight full vertices) first.  The
// host counted them (struct Brick); a list that would pass its count is cut, and *bad is set.
__global__ void __launch_bounds__(256) k_build_bricks(int nx, int ny, int nz, double sT, double dS, double C,
                                                      const float4 *rec, const Brick *bricks, BrickLists out, int *bad)
{
    __shared__ int wsum[2][8], base[2];
    __shared__ bool full_at[kLat];
    const Brick B = bricks[blockIdx.x];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    // ranks of up to 256 entries of two kinds, in thread order; returns the rank in the entry's own kind
    auto ranks = [&](bool k0, bool k1) {
        const unsigned b0 = __ballot_sync(kFull, k0), b1 = __ballot_sync(kFull, k1), lt = (1u << lane) - 1u;
        if (lane == 0) { wsum[0][wid] = __popc(b0); wsum[1][wid] = __popc(b1); }
        __syncthreads();
        const int k = k1 ? 1 : 0;
        int r = base[k] + __popc((k ? b1 : b0) & lt);
        for (int i = 0; i < wid; ++i) r += wsum[k][i];
        __syncthreads();
        if (threadIdx.x < 2) for (int i = 0; i < 8; ++i) base[threadIdx.x] += wsum[threadIdx.x][i];
        __syncthreads();
        return r;
    };
    if (threadIdx.x < 2) base[threadIdx.x] = 0;
    __syncthreads();
    const int nl = kLatX * kLatY * (B.planes + 1);
    for (int l0 = 0; l0 < nl; l0 += 256) {
        const int l = l0 + threadIdx.x, lx = l % kLatX, ly = (l / kLatX) % kLatY, lz = l / (kLatX * kLatY);
        const int X = B.x0 + lx, J = B.y0 + ly, K = B.z0 + lz;
        const bool in = l < nl && X <= nx && J <= ny;
        int cnt[3], cntd[3], nT = 0, nB;
        double M[6];
        bool T[2][2][2], Td[2][2][2];
        if (in) vertex_static(nx, ny, nz, rec, X, J, K, cnt, nT, M, T, cntd, nB, Td);
        const bool full = in && nT == 8, part = in && nT > 0 && nT < 8;
        if (l < kLat) full_at[l] = full;
        const int r = ranks(full, part);
        if (full || part) {
            const int at = full ? r : B.nfull + r;
            if (at >= (full ? B.nfull : B.nvert)) { *bad = 1; continue; }
            const double r0 = cnt[0] ? 1.0 / cnt[0] : 0.0, r1 = cnt[1] ? 1.0 / cnt[1] : 0.0,
                         r2 = cnt[2] ? 1.0 / cnt[2] : 0.0, iso = sT * nT;
            out.vloc[B.vbase + at] = (unsigned short)(lx | ly << 5 | lz << 9);
            out.k4[B.vbase + at] = make_float4((float)(C * r0 * r0 * (iso + dS * M[0])), (float)(C * r1 * r1 * (iso + dS * M[1])),
                                               (float)(C * r2 * r2 * (iso + dS * M[2])), (float)(C * r0 * r1 * dS * M[3]));
            out.k2[B.vbase + at] = make_float2((float)(C * r0 * r2 * dS * M[4]), (float)(C * r1 * r2 * dS * M[5]));
            if (part) {   // valid pairs: bit 4 a + o1 + 2 o2 as in the sweep
                unsigned w = 0;
                for (int o2 = 0; o2 < 2; ++o2)
                    for (int o1 = 0; o1 < 2; ++o1) {
                        const int o = o1 + 2 * o2;
                        if (T[o2][o1][0] && T[o2][o1][1]) w |= 1u << o;
                        if (T[o2][0][o1] && T[o2][1][o1]) w |= 16u << o;
                        if (T[0][o2][o1] && T[1][o2][o1]) w |= 256u << o;
                    }
                out.vpair[B.pbase + r] = (unsigned short)w;
            }
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && (base[0] != B.nfull || base[0] + base[1] != B.nvert)) *bad = 1;
    if (threadIdx.x < 2) base[threadIdx.x] = 0;
    __syncthreads();
    const int no = 32 * kBrickY * B.planes;
    auto tissue = [&](int i, int j, int k) {
        return i >= 0 && j >= 0 && k >= 0 && i < nx && j < ny && k < nz &&
               rec_tissue(rec[i + (long long)nx * (j + (long long)ny * k)]);
    };
    for (int o0 = 0; o0 < no; o0 += 256) {
        const int o = o0 + threadIdx.x, ox = o & 31, oy = (o >> 5) % kBrickY, oz = (o >> 5) / kBrickY;
        const int i = B.x0 + ox, j = B.y0 + oy, k = B.z0 + oz;
        const bool t = o < no && ox < kBrickX && tissue(i, j, k);
        bool inner = t;
        if (t)
            for (int v = 0; v < 8; ++v) inner = inner && full_at[ox + (v & 1) + kLatX * (oy + ((v >> 1) & 1) + kLatY * (oz + (v >> 2)))];
        const int r = ranks(inner, t && !inner);
        if (t) {
            const int at = inner ? r : B.ninner + r;
            if (at >= (inner ? B.ninner : B.nout)) { *bad = 1; continue; }
            out.out[B.obase + at] = make_float2(rec[i + (long long)nx * (j + (long long)ny * k)].w,
                                                __int_as_float(ox | oy << 5 | oz << 9));
            if (!inner)
                out.oflag[B.fbase + r] = (unsigned char)(tissue(i - 1, j, k) | tissue(i + 1, j, k) << 1 |
                                                         tissue(i, j - 1, k) << 2 | tissue(i, j + 1, k) << 3 |
                                                         tissue(i, j, k - 1) << 4 | tissue(i, j, k + 1) << 5);
        }
    }
    __syncthreads();
    if (threadIdx.x == 0 && (base[0] != B.ninner || base[0] + base[1] != B.nout)) *bad = 1;
}

}  // namespace gbep
