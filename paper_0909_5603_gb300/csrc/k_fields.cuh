// k_fields.cuh -- device functions of the grid phases (cell addressing, the absorbing
// layer, the fused Yee update, the fixed-pass filter sweeps, the periodic ghost copy),
// shared by the per-phase kernels of k_fields.cu and the persistent batched step.
#pragma once
#include "pic_internal.h"

namespace pic {

struct CellPos {
    int ii;       // instance
    int i, j, k;  // interior cell
    long long p;  // padded linear index
};

__device__ __forceinline__ bool cell_of(const Launch &L, long long g, CellPos &c, const InstDev *&I)
{
    if (g >= L.total_cells) return false;
    c.ii = find_instance_ll(L.cell_start, L.ninst, g);
    I = L.inst + c.ii;
    const int r = (int)(g - L.cell_start[c.ii]);  // < 2^31 cells per instance
    const int rq = fast_div(r, I->div_n0);
    c.i = r - rq * I->n[0];
    c.k = fast_div(rq, I->div_n1);
    c.j = rq - c.k * I->n[1];
    c.p = (c.i + I->gh[0]) + I->sy * (c.j + I->gh[1]) + I->sz * (c.k + I->gh[2]);
    return true;
}

// Offsets to the +1 / -1 neighbour along each axis (0 on an inactive axis).
__device__ __forceinline__ void neighbour_offsets(const InstDev &I, const CellPos &c, long long up[3], long long dn[3])
{
    const long long st[3] = {1, I.sy, I.sz};
    const int idx[3] = {c.i, c.j, c.k};
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        if (I.ndim == 2 && a == 1) {
            up[a] = dn[a] = 0;
            continue;
        }
        const bool per = I.bc[a] == 0;
        up[a] = (per && idx[a] == I.n[a] - 1) ? -(long long)(I.n[a] - 1) * st[a] : st[a];
        dn[a] = (per && idx[a] == 0) ? (long long)(I.n[a] - 1) * st[a] : -st[a];
    }
}

// Absorbing-layer factor prod_a (1 - s (d_a / L)^2), d_a = depth into the layer, read
// from the per-axis tables the host filled in FP64 (product taken x, y, z in order).
template <typename R>
__device__ __forceinline__ R damp_factor(const InstDev &I, const CellPos &c)
{
    R f = R(1);
    const int idx[3] = {c.i, c.j, c.k};
#pragma unroll
    for (int a = 0; a < 3; ++a)
        if (I.damp[a]) f *= ((const R *)I.damp[a])[idx[a]];
    return f;
}

// The whole Yee update of a step in one kernel (Yee solver, no antenna): B half step, E
// step, damped B half step.  It reads E^n, B^n and J once and writes E^{n+1}, B^{n+1}
// once (60 bytes per cell in FP32 instead of 120 for the three-kernel sequence).  The
// inputs are the current E / B buffer pair and the outputs go to the other one (*fpar
// flips after the last CTA), so no CTA overwrites a value that a neighbouring CTA still
// reads.  A cell near a periodic face is also stored at its images in the ghost layers
// beyond the opposite faces (what the gather's TMA boxes read there), instead of one ghost
// copy launch per periodic axis.
//
// A warp is one row of 32 columns along x, a thread one column, and the block marches
// along z through a chunk of tz planes.  In 3D its NW warps are NW rows along y; the outer
// column and rows (one below, two above) only feed their neighbours, so a block puts out
// 29 x (NW - 3) columns.  In 2D3V every warp marches alone through its own strip and chunk.  At
// plane i a thread forms, of its own column,
//   B^{n+1/2}(i+2) = B^n - dt/2 curl E^n            (E^n of planes i+2, i+3)
//   E^{n+1}(i+1)  = f (E^n + dt (curl B^{n+1/2} - J))  (B^{n+1/2} of planes i, i+1)
//   B^{n+1}(i)    = f (B^{n+1/2} - dt/2 curl E^{n+1})  (E^{n+1} of planes i, i+1)
// with the planes in registers, the x neighbours by shuffles and only the y neighbours
// through shared memory, all of them formed at earlier planes: one block barrier per plane
// (none in 2D3V).  The planes to come are copied (cp.async) into a ring of kMxAhead planes in
// shared memory, every thread its own column, so their latency costs no registers.
// Outside an absorbing box every field is zero; periodic axes wrap.  Each value is formed
// by the same expression as in k_bhalf / k_efull.
//
// It is bound by instruction issue (67 %) together with the latency of each plane's chain.
// Against a thread per column of 32 x 8 with all neighbours in shared memory, two barriers
// and the next plane's loads in registers, per step: 128x128x1024 380 -> 344 us (1.0 GB, 44 %
// of the copy rate), 64^3 periodic 37 -> 24, 32x32x256 29 -> 23, 48x48x128 FP64 90 -> 75,
// 128x128 2D3V 18 -> 9.4, a batch of 32 2D3V instances 108 -> 40 us.
constexpr int kMxCols = 29;  // columns along x that a warp puts out

template <typename R>
__host__ __device__ constexpr int mx_ahead()
{
    return sizeof(R) == 4 ? 4 : 3;
}

// the ring (nine components a plane) and, in 3D, rows of y neighbours: two planes of six
// components
template <typename R, int ND, int NW>
constexpr size_t maxwell_fused_smem()
{
    return sizeof(R) * 32 * NW * (9 * mx_ahead<R>() + (ND == 3 ? 2 * 6 : 0));
}

// cp.async of one value, or a zero
template <typename R>
__device__ __forceinline__ void mx_copy(R *dst, const R *src, bool ok)
{
    const unsigned d = static_cast<unsigned>(__cvta_generic_to_shared(dst));
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;\n" ::"r"(d), "l"(src), "n"(sizeof(R)),
                 "r"(ok ? (int)sizeof(R) : 0)
                 : "memory");
}

// index along one axis of the cell at q: false outside an absorbing box; wrapped on a
// periodic axis
__device__ __forceinline__ bool mx_axis(int q, int n, int bc, int &w)
{
    if (q >= 0 && q < n) {
        w = q;
        return true;
    }
    if (bc != 0) return false;
    w = ((q % n) + n) % n;
    return true;
}

// Block g of the launch's tiles (tile_start: the instances' first tiles), by NW warps.
// tz: planes per chunk (0: the instance's own, mx_planes).  images: also store the periodic
// images of the cells.
template <typename R, int ND, int NW>
__device__ __forceinline__ void maxwell_fused_block(const Launch &L, const long long *tile_start, int filtered,
                                                    const long long g, int tz, bool images)
{
    constexpr unsigned kAll = 0xffffffffu;
    constexpr int TY = NW - 3, NT = 32 * NW;
    extern __shared__ __align__(16) unsigned char msm[];
    constexpr int D = mx_ahead<R>();
    R *ring = (R *)msm;         // [plane % D][E of the plane, B of the one before, J of the one before that][thread]
    R *sm = ring + 9 * D * NT;  // [plane parity][Ex Ez Bx Bz Ex' Ez'][row][32]
    if (g >= tile_start[L.ninst]) return;
    const int ii = find_instance_ll(tile_start, L.ninst, g);
    const InstDev &I = L.inst[ii];
    const int n0 = I.n[0], n1 = I.n[1], n2 = I.n[2];
    // (the shuffle tells the compiler that the warp's number, and with it its planes, is the
    // same in all lanes)
    const int lane = threadIdx.x & 31, row = __shfl_sync(kAll, (int)(threadIdx.x >> 5), 0);
    if (tz == 0) tz = I.mx_planes;
    const int ntx = (n0 + kMxCols - 1) / kMxCols;
    long long r = g - tile_start[ii];
    if (ND == 2) r = r * NW + row;  // this warp's strip and chunk
    const int x0 = (int)(r % ntx) * kMxCols;
    r /= ntx;
    int y0 = 0;
    if (ND == 3) {
        const int nty = (n1 + TY - 1) / TY;
        y0 = (int)(r % nty) * TY;
        r /= nty;
    }
    const int z0 = (int)r * tz;
    if (z0 >= n2) return;  // (2D3V: a warp beyond the last strip)
    const int z1 = min(z0 + tz, n2);
    const int par = *(volatile const int *)I.fpar;
    // the components of each field are cstride elements apart
    const long long cs = I.cstride;
    const int nsweeps = I.filter_passes > 0 ? (I.ndim == 3 ? 3 : 2) : 0;
    const R *Ein = (const R *)(par ? I.E2[0] : I.E[0]), *Bin = (const R *)(par ? I.B2[0] : I.B[0]);
    R *Eout = (R *)(par ? I.E[0] : I.E2[0]), *Bout = (R *)(par ? I.B[0] : I.B2[0]);
    const R *Jin = (const R *)((filtered && (nsweeps & 1)) ? I.Jt[0] : I.J[0]);
    const StepCoef<R> &K = coef<R>(I);
    const R h = K.half_dt, dt = K.dt;
    const R ix = K.inv_dx[0], iy = K.inv_dx[1], iz = K.inv_dx[2];
    const R *dampx = (const R *)I.damp[0], *dampy = (const R *)I.damp[1], *dampz = (const R *)I.damp[2];
    // this thread's column: its padded in-plane offset, whether it lies in the box, its x
    // and y damping factors multiplied in the order of damp_factor
    const int xc = x0 - 1 + lane, yc = ND == 3 ? y0 - 1 + row : 0;
    int x = 0, y = 0;
    bool in = mx_axis(xc, n0, I.bc[0], x);
    if (ND == 3) in = mx_axis(yc, n1, I.bc[1], y) && in;
    const unsigned off = (unsigned)(x + I.gh[0]) + (unsigned)I.sy * (unsigned)(y + I.gh[1]);  // < 2^31: one plane
    R fxy = R(1);
    if (in && dampx) fxy *= dampx[x];
    if (in && ND == 3 && dampy) fxy *= dampy[y];
    // whether it is put out here, and where its images lie in the ghost layers of periodic
    // axes: bit 0 (1) of mx when x is within the ghost width of the lower (upper) face, my for y
    const bool tok = lane >= 1 && lane <= kMxCols && xc < n0 && (ND == 2 || (row >= 1 && row <= TY && yc < n1));
    const int mx = images && I.bc[0] == 0 ? (xc < I.gh[0] ? 1 : 0) | (xc >= n0 - I.gh[0] ? 2 : 0) : 0;
    const int my = ND == 3 && images && I.bc[1] == 0 ? (yc < I.gh[1] ? 1 : 0) | (yc >= n1 - I.gh[1] ? 2 : 0) : 0;
    // what the planes need of the instance, kept in registers (its device copy would be read
    // again after every store)
    const bool per2 = I.bc[2] == 0, zimg = images && per2;
    const long long sy = I.sy, sz = I.sz;
    const int gh2 = I.gh[2];
    // z: padded offset of plane k (-1 <= k <= n2 + 2: at most one wrap), false outside an
    // absorbing box
    auto zplane = [&](int k, long long &zo) -> bool {
        const int z = k < 0 ? k + n2 : k >= n2 ? k - n2 : k;
        zo = sz * (long long)(z + gh2);
        return per2 || z == k;
    };
    // plane n of the ring: E^n(n), B^n(n-1), J(n-2), as far as the chunk needs them
    auto fetch = [&](int n) {
        R *d = ring + (unsigned)(n - z0) % D * 9 * NT + threadIdx.x;
        auto copy3 = [&](const R *F, int k, R *to, bool wanted) {
            if (!wanted) return;
            long long zo;
            const bool ok = zplane(k, zo) && in;
            const R *plane = F + zo;  // (off lies in the plane, whether copied or not)
            mx_copy(to, plane + off, ok);
            mx_copy(to + NT, plane + cs + off, ok);
            mx_copy(to + 2 * NT, plane + 2 * cs + off, ok);
        };
        copy3(Ein, n, d, n <= z1 + 2);
        copy3(Bin, n - 1, d + 3 * NT, n - 1 <= z1);
        copy3(Jin, n - 2, d + 6 * NT, n - 2 >= z0 && n - 2 <= z1);
        asm volatile("cp.async.commit_group;\n" ::: "memory");
    };
    const int at = threadIdx.x, up = min(row + 1, NW - 1) * 32 + lane, dn = max(row - 1, 0) * 32 + lane;

    R e1[3] = {}, e2[3], h0[3] = {}, h1[3] = {}, q0[3] = {}, f0 = R(1);
#pragma unroll
    for (int n = 0; n < D; ++n) fetch(z0 + n);
    {
        long long zo;
        const bool ok = zplane(z0 - 1, zo) && in;
#pragma unroll
        for (int c = 0; c < 3; ++c) e2[c] = ok ? (Ein + c * cs + zo)[off] : R(0);
    }
    if (ND == 3) {
        R *s = sm + ((z0 - 3) & 1) * 6 * NT;
        s[at] = e2[0];
        s[NT + at] = e2[2];
        __syncthreads();
    }
#pragma unroll 1
    for (int i = z0 - 3; i < z1; ++i) {
        const R *s = sm + (i & 1) * 6 * NT;
        R *t = sm + ((i + 1) & 1) * 6 * NT;
        asm volatile("cp.async.wait_group %0;\n" ::"n"(D - 1) : "memory");
        R e3[3], b2[3], j1[3];
        {
            const R *d = ring + (unsigned)(i + 3 - z0) % D * 9 * NT + threadIdx.x;
#pragma unroll
            for (int c = 0; c < 3; ++c) {
                e3[c] = d[c * NT];
                b2[c] = d[(3 + c) * NT];
                j1[c] = d[(6 + c) * NT];
            }
        }
        fetch(i + 3 + D);  // in the place of the plane just taken
        long long zo;
        R h2[3] = {R(0), R(0), R(0)}, q1[3] = {R(0), R(0), R(0)}, f1 = fxy;
        if (i + 2 <= z1) {
            const R ex = e2[0], ey = e2[1], ez = e2[2];
            R dEz_dy = R(0), dEx_dy = R(0);
            const R dEy_dz = (e3[1] - ey) * iz;
            const R dEx_dz = (e3[0] - ex) * iz;
            const R dEz_dx = (__shfl_down_sync(kAll, ez, 1) - ez) * ix;
            const R dEy_dx = (__shfl_down_sync(kAll, ey, 1) - ey) * ix;
            if (ND == 3) {
                dEz_dy = (s[NT + up] - ez) * iy;
                dEx_dy = (s[up] - ex) * iy;
            }
            if (zplane(i + 2, zo) && in) {
                h2[0] = b2[0] - h * (dEz_dy - dEy_dz);
                h2[1] = b2[1] - h * (dEx_dz - dEz_dx);
                h2[2] = b2[2] - h * (dEy_dx - dEx_dy);
            }
        }
        if (i + 1 >= z0) {
            const R bx = h1[0], by = h1[1], bz = h1[2];
            R dBz_dy = R(0), dBx_dy = R(0);
            const R dBy_dz = (by - h0[1]) * iz, dBx_dz = (bx - h0[0]) * iz;
            const R dBz_dx = (bz - __shfl_up_sync(kAll, bz, 1)) * ix, dBy_dx = (by - __shfl_up_sync(kAll, by, 1)) * ix;
            if (ND == 3) {
                dBz_dy = (bz - s[3 * NT + dn]) * iy;
                dBx_dy = (bx - s[2 * NT + dn]) * iy;
            }
            if (zplane(i + 1, zo) && in) {
                const R f = dampz ? fxy * dampz[i + 1] : fxy;  // (an axis with a layer does not wrap)
                f1 = f;
                q1[0] = f * (e1[0] + dt * ((dBz_dy - dBy_dz) - j1[0]));
                q1[1] = f * (e1[1] + dt * ((dBx_dz - dBz_dx) - j1[1]));
                q1[2] = f * (e1[2] + dt * ((dBy_dx - dBx_dy) - j1[2]));
            }
        }
        if (i >= z0) {
            const R ex = q0[0], ey = q0[1], ez = q0[2];
            R dEz_dy = R(0), dEx_dy = R(0);
            const R dEy_dz = (q1[1] - ey) * iz;
            const R dEx_dz = (q1[0] - ex) * iz;
            const R dEz_dx = (__shfl_down_sync(kAll, ez, 1) - ez) * ix;
            const R dEy_dx = (__shfl_down_sync(kAll, ey, 1) - ey) * ix;
            if (ND == 3) {
                dEz_dy = (s[5 * NT + up] - ez) * iy;
                dEx_dy = (s[4 * NT + up] - ex) * iy;
            }
            if (tok) {
                zo = sz * (long long)(i + gh2);
                R bx = h0[0] - h * (dEz_dy - dEy_dz);
                R by = h0[1] - h * (dEx_dz - dEz_dx);
                R bz = h0[2] - h * (dEy_dx - dEx_dy);
                bx *= f0;
                by *= f0;
                bz *= f0;
                auto store = [&](long long p, unsigned o) {  // p the same in the whole warp
                    (Bout + p)[o] = bx;
                    (Bout + cs + p)[o] = by;
                    (Bout + 2 * cs + p)[o] = bz;
                    (Eout + p)[o] = ex;
                    (Eout + cs + p)[o] = ey;
                    (Eout + 2 * cs + p)[o] = ez;
                };
                // the cell (0) and its images + n (1) and - n (2): along z and y the same for
                // the whole warp, along x for the lanes near a face
                const int mz = zimg ? (i < gh2 ? 1 : 0) | (i >= n2 - gh2 ? 2 : 0) : 0;
#pragma unroll 1
                for (int az = 0; az <= mz; ++az) {
                    if (az && !(mz & az)) continue;
                    const long long pz = zo + sz * (long long)(az == 1 ? n2 : az == 2 ? -n2 : 0);
#pragma unroll 1
                    for (int ay = 0; ay <= my; ++ay) {
                        if (ay && !(my & ay)) continue;
                        const long long p = pz + sy * (long long)(ay == 1 ? n1 : ay == 2 ? -n1 : 0);
                        store(p, off);
                        if (mx & 1) store(p, off + (unsigned)n0);
                        if (mx & 2) store(p, off - (unsigned)n0);
                    }
                }
            }
        }
        if (ND == 3) {
            t[at] = e3[0];
            t[NT + at] = e3[2];
            t[2 * NT + at] = h2[0];
            t[3 * NT + at] = h2[2];
            t[4 * NT + at] = q1[0];
            t[5 * NT + at] = q1[2];
            __syncthreads();
        }
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            e1[c] = e2[c];
            e2[c] = e3[c];
            h0[c] = h1[c];
            h1[c] = h2[c];
            q0[c] = q1[c];
        }
        f0 = f1;
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");  // (only empty groups are left)
}

// Binomial filter along one axis, all passes at once.  The x, y and z operators (each
// with its boundary: periodic wrap, or zero outside an absorbing box after every pass)
// act on different axes and commute, so `passes` rounds of (x, y, z) equal x^passes,
// y^passes, z^passes.  One CTA takes a pencil of kPencil cells along the axis (times 32
// x-columns for the y and z axes), loads it with `passes` halo cells per side into shared
// memory, applies the passes there (J <- J(i-1)/4 + J(i)/2 + J(i+1)/4, re-zeroing cells
// outside an absorbing box after each pass) and writes the pencil back: one read and one
// write per cell and axis instead of one per pass.  Reads src, writes dst (J / Jt).
constexpr int kPencil = 64;
constexpr int kMaxPasses = 8;

__device__ __forceinline__ bool filter_active_axis(const InstDev &I, int axis)
{
    return I.filter_passes > 0 && !(I.ndim == 2 && axis == 1);
}

// The same filter with the number of passes P known at compile time (P <= 4, every
// instance of the launch alike), in registers, without shared memory or barriers, on the
// pencils of k_filter_axis.  Binomial weight C(2P, m) / 4^P of tap m (exact in FP32).
__host__ __device__ constexpr double binomial_weight(int P, int m)
{
    double c = 1.0;
    for (int t = 1; t <= m; ++t) c = c * (2 * P - t + 1) / t;
    return c / (double)(1 << (2 * P));
}

// The cell whose value stands at q along an axis of n cells for the convolution (negated
// when it returns -1, nothing there when it returns 0):
// the wrapped cell on a periodic axis; beyond an absorbing face the odd reflection about
// the first node outside.  P passes of 1-2-1 with that node and all beyond it zeroed after
// each pass equal one convolution of the field continued that way (the reflection
// principle: the continued field stays odd about the node, which therefore stays zero,
// under every pass; a window of P <= 4 < n cells meets one face only), so no cell needs the
// passes one by one.  Nothing: the node itself, or past the cells that count.
__device__ __forceinline__ int filter_source(int &q, int n, int P, bool per)
{
    if (q >= 0 && q < n) return 1;
    if (per) {
        q = ((q % n) + n) % n;  // (a ragged last pencil can reach more than one period past the end)
        return 1;
    }
    if (q == -1 || q == n || q >= n + P) return 0;
    q = q < 0 ? -2 - q : 2 * n - q;
    return -1;
}

// v, negated when neg.  FP64: in the sign bit, as the FP64 pipe, which a select between v and
// -v goes through, bounds the filter there (64x64x128 periodic cells, one pass: 58 us
// with the select, 53 without any).
__device__ __forceinline__ float negate_if(float v, bool neg) { return neg ? -v : v; }
__device__ __forceinline__ double negate_if(double v, bool neg)
{
    return __hiloint2double(__double2hiint(v) ^ (neg ? (int)0x80000000 : 0), __double2loint(v));
}

// y and z axes: lane = x column (coalesced), each warp takes kPencil / 8 consecutive
// cells along the axis and loads them with P halo cells per side into registers
// (filter_source); the outputs are (2P+1)-tap convolutions.  Four blocks of 64 registers per
// SM in FP32 hide the loads better than three of 80, also with the spills of the blocks at
// the faces (100 bytes with three passes, 204 with four; all axes of 128x128x256 cells with
// four passes: 99 us periodic and 99 absorbing, 127 and 137 before).
template <typename R, int P>
__device__ __forceinline__ void filter_col_block(const Launch &L, int axis, const long long *pencil_start, int src_is_jt,
                                                 const long long g)
{
    constexpr int S = kPencil / 8;
    constexpr int W = S + 2 * P;
    if (g >= pencil_start[L.ninst]) return;
    const int ii = find_instance_ll(pencil_start, L.ninst, g);
    const InstDev &I = L.inst[ii];
    if (!filter_active_axis(I, axis)) return;
    const int n = I.n[axis];
    const bool per = I.bc[axis] == 0;
    const int nseg = (n + kPencil - 1) / kPencil;
    long long r = g - pencil_start[ii];
    const int qs = (int)(r % nseg) * kPencil + (threadIdx.x >> 5) * S;  // this thread's first cell
    r /= nseg;
    const int ncol = (I.n[0] + 31) / 32;
    const int x = (int)(r % ncol) * 32 + (threadIdx.x & 31);
    const int other = (int)(r / ncol);  // z for the y axis, y for the z axis
    if (x >= I.n[0] || qs >= n) return;
    const long long sa = axis == 1 ? I.sy : I.sz;
    const long long lo = axis == 1 ? (x + I.gh[0]) + I.sy * I.gh[1] + I.sz * (long long)(other + I.gh[2])
                                   : (x + I.gh[0]) + I.sy * (long long)(other + I.gh[1]) + I.sz * I.gh[2];
    const bool inside = qs - P >= 0 && qs + S + P <= n;
    void *const *src = src_is_jt ? I.Jt : I.J;
    void *const *dst = src_is_jt ? I.J : I.Jt;
    // all three windows first (the source and destination arrays differ)
    R win[3][W];
    if (inside) {
#pragma unroll
        for (int comp = 0; comp < 3; ++comp) {
            const R *__restrict__ a = (const R *)src[comp];
#pragma unroll
            for (int m = 0; m < W; ++m) win[comp][m] = a[lo + (long long)(qs - P + m) * sa];
        }
    } else {
        int at[W];
        unsigned ok = 0, neg = 0;
#pragma unroll
        for (int m = 0; m < W; ++m) {
            at[m] = qs - P + m;
            const int f = filter_source(at[m], n, P, per);
            ok |= f != 0 ? 1u << m : 0u;
            neg |= f < 0 ? 1u << m : 0u;
        }
#pragma unroll
        for (int comp = 0; comp < 3; ++comp) {
            const R *__restrict__ a = (const R *)src[comp];
#pragma unroll
            for (int m = 0; m < W; ++m) win[comp][m] = (ok >> m) & 1u ? a[lo + (long long)at[m] * sa] : R(0);
        }
        if (neg) {
#pragma unroll
            for (int comp = 0; comp < 3; ++comp)
#pragma unroll
                for (int m = 0; m < W; ++m)
                    win[comp][m] = negate_if(win[comp][m], (neg >> m) & 1u);
        }
    }
#pragma unroll
    for (int comp = 0; comp < 3; ++comp) {
        R *__restrict__ b = (R *)dst[comp];
#pragma unroll
        for (int t = 0; t < S; ++t) {
            R v = R(0);
#pragma unroll
            for (int m = 0; m <= 2 * P; ++m) v += R(binomial_weight(P, m)) * win[comp][t + m];
            if (qs + t < n) b[lo + (long long)(qs + t) * sa] = v;
        }
    }
}

// x axis: warp w takes rows w, w + 8, w + 16, w + 24 of the pencil.  It first loads the
// kPencil + 2P window of all three components of all four rows into registers
// (coalesced, all in flight together), then per row stores the window into its own
// slice of shared memory (warp-synchronous, no block barrier) and each lane forms two
// outputs from it, convolutions over the window (filter_source).  (With the passes run one
// by one in the lanes near an absorbing face, beside the convolution of the others, the
// three axes took 201 us instead of 89 for 48x48x128 FP64 cells, and 382 instead of 324 us
// for 128x128x1024 FP32 ones.)
// sw: shared memory for the windows, 8 x 3 x (kPencil + 2P) values
template <typename R, int P>
__device__ __forceinline__ void filter_row_block(const Launch &L, const long long *pencil_start, int src_is_jt,
                                                 const long long g, R *sw)
{
    constexpr int W = kPencil + 2 * P;
    if (g >= pencil_start[L.ninst]) return;
    const int ii = find_instance_ll(pencil_start, L.ninst, g);
    const InstDev &I = L.inst[ii];
    if (!filter_active_axis(I, 0)) return;
    const int n = I.n[0];
    const bool per = I.bc[0] == 0;
    const int nseg = (n + kPencil - 1) / kPencil;
    long long r = g - pencil_start[ii];
    const int q0 = (int)(r % nseg) * kPencil;
    r /= nseg;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const bool inside = q0 - P >= 0 && q0 + kPencil + P <= n;
    void *const *src = src_is_jt ? I.Jt : I.J;
    void *const *dst = src_is_jt ? I.J : I.Jt;
    R(*win)[W] = reinterpret_cast<R(*)[W]>(sw + warp * 3 * W);
    constexpr int NR = 4, NC = (W + 31) / 32;  // rows per warp, window chunks of 32
    const long long nrows = (long long)I.n[1] * I.n[2];
    long long lo[NR];
    R pre[NR][3][NC];
    // this lane's window cells (the same in every row)
    int qi[NC];
    bool qok[NC], qneg[NC];
#pragma unroll
    for (int c = 0; c < NC; ++c) {
        const int i = 32 * c + lane;
        int q = q0 - P + i;
        const int f = i < W ? (inside ? 1 : filter_source(q, n, P, per)) : 0;
        qi[c] = q;
        qok[c] = f != 0;
        qneg[c] = f < 0;
    }
#pragma unroll
    for (int j = 0; j < NR; ++j) {
        const long long row = r * 32 + warp + 8 * j;
        const bool rok = row < nrows;
        const int y = rok ? (int)(row % I.n[1]) : 0, z = rok ? (int)(row / I.n[1]) : 0;
        lo[j] = I.gh[0] + I.sy * (long long)(y + I.gh[1]) + I.sz * (long long)(z + I.gh[2]);
#pragma unroll
        for (int comp = 0; comp < 3; ++comp)
#pragma unroll
            for (int c = 0; c < NC; ++c)
                pre[j][comp][c] = (rok && qok[c]) ? ((const R *)src[comp])[lo[j] + qi[c]] : R(0);
    }
#pragma unroll
    for (int j = 0; j < NR; ++j) {
        if (r * 32 + warp + 8 * j >= nrows) break;
#pragma unroll
        for (int comp = 0; comp < 3; ++comp)
#pragma unroll
            for (int c = 0; c < NC; ++c)
                if (32 * c + lane < W) win[comp][32 * c + lane] = negate_if(pre[j][comp][c], qneg[c]);
        __syncwarp();
#pragma unroll
        for (int h = 0; h < 2; ++h) {
            const int t = lane + 32 * h;  // output q0 + t, window cells t .. t + 2P
            const int q = q0 + t;
            if (q >= n) continue;
#pragma unroll
            for (int comp = 0; comp < 3; ++comp) {
                R v = R(0);
#pragma unroll
                for (int m = 0; m <= 2 * P; ++m) v += R(binomial_weight(P, m)) * win[comp][t + m];
                ((R *)dst[comp])[lo[j] + q] = v;
            }
        }
        __syncwarp();  // the window is rewritten for the next row
    }
}

// Periodic ghost exchange of the six E/B components along one axis (after the whole
// step); ghosts of earlier axes are included so corners come out right.
// Element r of the ghost copy of instance I along `axis` (0 <= r < ghost_elems(I, axis)).
template <typename R>
__device__ __forceinline__ void ghost_elem(const InstDev &I, int axis, long long r)
{
    // ghost slab: 2*gh layers along `axis` x padded extents of the other two axes
    const int gh = I.gh[axis];
    const int o1 = axis == 0 ? 1 : 0, o2 = axis == 2 ? 1 : 2;
    const long long e1 = I.P[o1], e2 = I.P[o2];
    const long long slab = 2LL * gh * e1 * e2;
    if (r >= 6 * slab) return;
    const int comp = (int)(r / slab);
    r -= comp * slab;
    const int layer = (int)(r % (2 * gh));
    r /= 2 * gh;
    const long long a1 = r % e1, a2 = r / e1;
    const int n = I.n[axis];
    // destination padded coordinate along axis and its periodic source
    const int dpos = layer < gh ? layer : gh + n + (layer - gh);
    const int spos = layer < gh ? dpos + n : dpos - n;
    long long st[3] = {1, I.sy, I.sz};
    const long long base = a1 * st[o1] + a2 * st[o2];
    R *f = (R *)eb_field(I, comp);
    f[base + dpos * st[axis]] = f[base + spos * st[axis]];
}

// Elements of the ghost copy of instance I along `axis` (0 when the axis is not periodic).
__device__ __forceinline__ long long ghost_elems(const InstDev &I, int axis)
{
    if (I.bc[axis] != 0 || (I.ndim == 2 && axis == 1)) return 0;
    const int o1 = axis == 0 ? 1 : 0, o2 = axis == 2 ? 1 : 2;
    return 6LL * 2 * I.gh[axis] * I.P[o1] * I.P[o2];
}

}  // namespace pic
