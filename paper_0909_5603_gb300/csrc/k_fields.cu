// k_fields.cu -- grid kernels of the boosted-frame PIC step on sm_103a: Yee FDTD
// half/whole updates with the absorbing layer, binomial current filter sweeps, periodic
// ghost exchange for the TMA gather boxes, and the FP64 field reductions / read-outs.
//
// All stencil kernels run one thread per interior cell of a flattened cell space over
// every instance of the launch (x fastest, so loads and stores coalesce along rows).
// Neighbours along periodic axes wrap by index; along absorbing axes they read the
// zero ghost layers.
#include "k_fields.cuh"

#include <algorithm>

namespace pic {

// Forward difference of F along axis a at padded index p, averaged over the two
// transverse axes with weights 7/12 (itself), 1/12 (edge neighbours), 1/48 (corners);
// up / dn are the +1 / -1 neighbour offsets of the cell (wrapping on periodic axes, 0 on
// an invariant one).
template <typename R>
__device__ __forceinline__ R ck_diff(const R *F, long long p, const long long up[3], const long long dn[3], int a)
{
    const int b = (a + 1) % 3, c = (a + 2) % 3;
    const long long ob[3] = {dn[b], 0, up[b]}, oc[3] = {dn[c], 0, up[c]};
    R sum = R(0);
#pragma unroll
    for (int ib = 0; ib < 3; ++ib)
#pragma unroll
        for (int ic = 0; ic < 3; ++ic) {
            const int edges = (ib != 1) + (ic != 1);
            const R w = edges == 0 ? R(7.0 / 12.0) : (edges == 1 ? R(1.0 / 12.0) : R(1.0 / 48.0));
            const long long q = p + ob[ib] + oc[ic];
            sum += w * (F[q + up[a]] - F[q]);
        }
    return sum;
}

// B <- B - (dt/2) curl E  [then x damping on the second half of the step].  CK: the
// low-dispersion differences (a template parameter, so that the Yee kernel keeps its
// small register footprint and full occupancy)
template <typename R, bool CK>
__global__ void __launch_bounds__(256) k_bhalf(Launch L, int damp)
{
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    CellPos c;
    const InstDev *Ip;
    if (!cell_of(L, g, c, Ip)) return;
    const InstDev &I = *Ip;
    long long up[3], dn[3];
    neighbour_offsets(I, c, up, dn);
    const EBPtr F = cur_eb(I);
    const R *Ex = (const R *)F.E[0], *Ey = (const R *)F.E[1], *Ez = (const R *)F.E[2];
    R *Bx = (R *)F.B[0], *By = (R *)F.B[1], *Bz = (R *)F.B[2];
    const StepCoef<R> &K = coef<R>(I);
    const R h = K.half_dt;
    const R ix = K.inv_dx[0], iy = K.inv_dx[1], iz = K.inv_dx[2];
    const long long p = c.p;
    R dEz_dy = R(0), dEy_dz, dEx_dz, dEz_dx, dEy_dx, dEx_dy = R(0);
    if (CK) {
        // low-dispersion solver: each forward difference averaged over its transverse
        // neighbours, 7/12 on itself, 1/12 on the edge and 1/48 on the corner ones (on
        // an invariant axis the neighbours are the cell itself)
        dEy_dz = ck_diff(Ey, p, up, dn, 2) * iz;
        dEx_dz = ck_diff(Ex, p, up, dn, 2) * iz;
        dEz_dx = ck_diff(Ez, p, up, dn, 0) * ix;
        dEy_dx = ck_diff(Ey, p, up, dn, 0) * ix;
        if (I.ndim == 3) {
            dEz_dy = ck_diff(Ez, p, up, dn, 1) * iy;
            dEx_dy = ck_diff(Ex, p, up, dn, 1) * iy;
        }
    } else {
        const R ex = Ex[p], ey = Ey[p], ez = Ez[p];
        dEy_dz = (Ey[p + up[2]] - ey) * iz;
        dEx_dz = (Ex[p + up[2]] - ex) * iz;
        dEz_dx = (Ez[p + up[0]] - ez) * ix;
        dEy_dx = (Ey[p + up[0]] - ey) * ix;
        if (I.ndim == 3) {
            dEz_dy = (Ez[p + up[1]] - ez) * iy;
            dEx_dy = (Ex[p + up[1]] - ex) * iy;
        }
    }
    R bx = Bx[p] - h * (dEz_dy - dEy_dz);
    R by = By[p] - h * (dEx_dz - dEz_dx);
    R bz = Bz[p] - h * (dEy_dx - dEx_dy);
    if (damp) {
        const R f = damp_factor<R>(I, c);
        bx *= f;
        by *= f;
        bz *= f;
    }
    Bx[p] = bx;
    By[p] = by;
    Bz[p] = bz;
}

// The low-dispersion half step of one 3D instance: a thread per column marches along z
// through tz planes (blockIdx.y) with its 3 x 3 neighbourhood of E on three planes in
// registers, so that a cell costs 27 loads of E instead of the 108 that k_bhalf's six
// differences ask for, which bound it there (addresses and L1, at 23 % of HBM).  The
// differences and their order are k_bhalf's.  128 registers, no spills, 16 warps an SM, and
// bound by the latency of a plane's loads; the three updates of a step: 64x64x512 162 -> 112
// us, 128x128x512 620 -> 395, 32x32x256 38 -> 33.  (Unrolled by three planes, so that none is
// moved: 140 us; with 96 registers 127.)
template <typename R>
__device__ __forceinline__ R ck_sum(const R d[9])
{
    R sum = R(0);
#pragma unroll
    for (int m = 0; m < 9; ++m) {
        const int edges = (m / 3 != 1) + (m % 3 != 1);
        const R w = edges == 0 ? R(7.0 / 12.0) : (edges == 1 ? R(1.0 / 12.0) : R(1.0 / 48.0));
        sum += w * d[m];
    }
    return sum;
}

// differences of the neighbourhood f[z][y][x] (entry 1 the cell itself), averaged as ck_diff
// does: its outer loop runs over axis a + 1, its inner one over axis a + 2
template <typename R, int A>
__device__ __forceinline__ R ck_diff3(const R (&f)[3][3][3])
{
    R d[9];
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int c = 0; c < 3; ++c)
            d[3 * b + c] = A == 0 ? f[c][b][2] - f[c][b][1] : (A == 1 ? f[b][2][c] - f[b][1][c] : f[2][c][b] - f[1][c][b]);
    return ck_sum(d);
}

__global__ void __launch_bounds__(128) k_bhalf_ck3(Launch L, int damp, int tz)
{
    using R = float;
    const InstDev &I = L.inst[0];
    const int n0 = I.n[0], n1 = I.n[1], n2 = I.n[2];
    const int col = blockIdx.x * 128 + threadIdx.x;
    if (col >= n0 * n1) return;
    CellPos c;
    c.ii = 0;
    c.j = fast_div(col, I.div_n0);
    c.i = col - c.j * n0;
    const EBPtr F = cur_eb(I);
    const StepCoef<R> &K = coef<R>(I);
    const R h = K.half_dt;
    const R ix = K.inv_dx[0], iy = K.inv_dx[1], iz = K.inv_dx[2];
    const long long sz = I.sz, base = (c.i + I.gh[0]) + I.sy * (c.j + I.gh[1]) + sz * I.gh[2];
    int off[3][3];  // of the neighbours in a plane, [y][x]
    {
        const int ox[3] = {I.bc[0] == 0 && c.i == 0 ? n0 - 1 : -1, 0, I.bc[0] == 0 && c.i == n0 - 1 ? 1 - n0 : 1};
        const int ny = n1 - 1, sy = (int)I.sy;
        const int oy[3] = {I.bc[1] == 0 && c.j == 0 ? ny * sy : -sy, 0, I.bc[1] == 0 && c.j == ny ? -ny * sy : sy};
#pragma unroll
        for (int y = 0; y < 3; ++y)
#pragma unroll
            for (int x = 0; x < 3; ++x) off[y][x] = oy[y] + ox[x];
    }
    const bool perz = I.bc[2] == 0;
    const R *const E[3] = {(const R *)F.E[0] + base, (const R *)F.E[1] + base, (const R *)F.E[2] + base};
    R *const B[3] = {(R *)F.B[0] + base, (R *)F.B[1] + base, (R *)F.B[2] + base};
    R f[3][3][3][3];  // [component][plane][y][x]
    auto load = [&](int k, int z) {
        const long long o = sz * (perz ? (k < 0 ? n2 - 1 : (k == n2 ? 0 : k)) : k);
#pragma unroll
        for (int m = 0; m < 3; ++m)
#pragma unroll
            for (int y = 0; y < 3; ++y)
#pragma unroll
                for (int x = 0; x < 3; ++x) f[m][z][y][x] = __ldg(E[m] + o + off[y][x]);
    };
    const int k0 = blockIdx.y * tz, k1 = min(k0 + tz, n2);
    load(k0 - 1, 0);
    load(k0, 1);
    for (c.k = k0; c.k < k1; ++c.k) {
        const long long o = sz * c.k;
        load(c.k + 1, 2);
        const R b0 = B[0][o], b1 = B[1][o], b2 = B[2][o];
        const R dEy_dz = ck_diff3<R, 2>(f[1]) * iz;
        const R dEx_dz = ck_diff3<R, 2>(f[0]) * iz;
        const R dEz_dx = ck_diff3<R, 0>(f[2]) * ix;
        const R dEy_dx = ck_diff3<R, 0>(f[1]) * ix;
        const R dEz_dy = ck_diff3<R, 1>(f[2]) * iy;
        const R dEx_dy = ck_diff3<R, 1>(f[0]) * iy;
        R bx = b0 - h * (dEz_dy - dEy_dz);
        R by = b1 - h * (dEx_dz - dEz_dx);
        R bz = b2 - h * (dEy_dx - dEx_dy);
        if (damp) {
            const R d = damp_factor<R>(I, c);
            bx *= d;
            by *= d;
            bz *= d;
        }
        B[0][o] = bx;
        B[1][o] = by;
        B[2][o] = bz;
#pragma unroll
        for (int m = 0; m < 3; ++m)
#pragma unroll
            for (int y = 0; y < 3; ++y)
#pragma unroll
                for (int x = 0; x < 3; ++x) {
                    f[m][0][y][x] = f[m][1][y][x];
                    f[m][1][y][x] = f[m][2][y][x];
                }
    }
}

// The fused Yee update (maxwell_fused_block).  The CTA of an
// instance that finishes last switches it to the buffer pair it wrote (every CTA has read
// the parity by then), so that no launch follows for it.
template <typename R, int ND>
__global__ void __launch_bounds__(32 * mx_warps<ND>(), mx_resident<R, ND>())
    k_maxwell_fused(Launch L, const long long *tile_start, int filtered)
{
    maxwell_fused_block<R, ND, mx_warps<ND>()>(L, tile_start, filtered, blockIdx.x, 0, true);
    __syncthreads();
    if (threadIdx.x == 0) {
        const int ii = find_instance_ll(tile_start, L.ninst, blockIdx.x);
        const InstDev &I = L.inst[ii];
        if (atomicAdd(I.mx_done, 1) == (int)(tile_start[ii + 1] - tile_start[ii]) - 1) {
            *I.mx_done = 0;
            *I.fpar ^= 1;
        }
    }
}

// E <- damping x (E + dt (curl B - J)), J = the filtered current of this step.
template <typename R>
__global__ void __launch_bounds__(256) k_efull(Launch L, int filtered)
{
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    CellPos c;
    const InstDev *Ip;
    if (!cell_of(L, g, c, Ip)) return;
    const InstDev &I = *Ip;
    long long up[3], dn[3];
    neighbour_offsets(I, c, up, dn);
    const EBPtr F = cur_eb(I);
    const R *Bx = (const R *)F.B[0], *By = (const R *)F.B[1], *Bz = (const R *)F.B[2];
    R *Ex = (R *)F.E[0], *Ey = (R *)F.E[1], *Ez = (R *)F.E[2];
    // one filter sweep per active axis alternates J -> Jt -> J ...
    const int nsweeps = I.filter_passes > 0 ? (I.ndim == 3 ? 3 : 2) : 0;
    void *const *Jsrc = (filtered && (nsweeps & 1)) ? I.Jt : I.J;
    const R *Jx = (const R *)Jsrc[0], *Jy = (const R *)Jsrc[1], *Jz = (const R *)Jsrc[2];
    const StepCoef<R> &K = coef<R>(I);
    const R dt = K.dt;
    const R ix = K.inv_dx[0], iy = K.inv_dx[1], iz = K.inv_dx[2];
    const long long p = c.p;
    const R bx = Bx[p], by = By[p], bz = Bz[p];
    R dBz_dy = R(0), dBy_dz = (by - By[p + dn[2]]) * iz, dBx_dz = (bx - Bx[p + dn[2]]) * iz;
    R dBz_dx = (bz - Bz[p + dn[0]]) * ix, dBy_dx = (by - By[p + dn[0]]) * ix, dBx_dy = R(0);
    if (I.ndim == 3) {
        dBz_dy = (bz - Bz[p + dn[1]]) * iy;
        dBx_dy = (bx - Bx[p + dn[1]]) * iy;
    }
    const R f = damp_factor<R>(I, c);
    Ex[p] = f * (Ex[p] + dt * ((dBz_dy - dBy_dz) - Jx[p]));
    Ey[p] = f * (Ey[p] + dt * ((dBx_dz - dBz_dx) - Jy[p]));
    Ez[p] = f * (Ez[p] + dt * ((dBy_dx - dBx_dy) - Jz[p]));
}

// A pencil is 32 lines parallel to `axis` times kPencil cells along it.  Lines: for the
// x axis, 32 consecutive (y, z) rows; for y and z, 32 consecutive x columns at one z (y).
// Work assignment without divisions: for the x axis a warp walks one line (lanes along x,
// coalesced), the 8 warps take lines 8 at a time; for y and z the lanes take the 32
// columns (coalesced along x) and the warps step along the axis.
template <typename R>
__global__ void __launch_bounds__(256) k_filter_axis(Launch L, int axis, const long long *pencil_start, int src_is_jt)
{
    __shared__ R buf[2][kPencil + 2 * kMaxPasses][33];
    __shared__ long long s_line[32];
    const long long g = blockIdx.x;
    if (g >= pencil_start[L.ninst]) return;
    const int ii = find_instance_ll(pencil_start, L.ninst, g);
    const InstDev &I = L.inst[ii];
    if (!filter_active_axis(I, axis)) return;
    const int P = min(I.filter_passes, kMaxPasses);
    const int n = I.n[axis];
    const bool per = I.bc[axis] == 0;
    const int nseg = (n + kPencil - 1) / kPencil;
    long long r = g - pencil_start[ii];
    const int q0 = (int)(r % nseg) * kPencil;  // first cell of the segment along the axis
    r /= nseg;
    const long long st[3] = {1, I.sy, I.sz};
    const long long sa = st[axis];
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    // line c -> padded offset of its cell 0 along the axis, or -1 when the line is absent
    if (tid < 32) {
        long long off = -1;
        const int c = tid;
        if (axis == 0) {
            const long long row = r * 32 + c;
            if (row < (long long)I.n[1] * I.n[2]) {
                const int y = (int)(row % I.n[1]), z = (int)(row / I.n[1]);
                off = I.gh[0] + st[1] * (y + I.gh[1]) + st[2] * (z + I.gh[2]);
            }
        } else {
            const int ncol = (I.n[0] + 31) / 32;
            const int x = (int)(r % ncol) * 32 + c;
            const int other = (int)(r / ncol);  // z for the y axis, y for the z axis
            if (x < I.n[0])
                off = axis == 1 ? (x + I.gh[0]) + st[1] * I.gh[1] + st[2] * (other + I.gh[2])
                                : (x + I.gh[0]) + st[1] * (other + I.gh[1]) + st[2] * I.gh[2];
        }
        s_line[c] = off;
    }
    __syncthreads();
    void *const *src = src_is_jt ? I.Jt : I.J;
    void *const *dst = src_is_jt ? I.J : I.Jt;
    const int len = kPencil + 2 * P;
    // (c, s) iteration: x axis: c = warp + 8 m, s = lane + 32 k; y, z: c = lane, s = warp + 8 k
    const int c_first = axis == 0 ? warp : lane, c_step = axis == 0 ? 8 : 32;
    const int s_first = axis == 0 ? lane : warp, s_step = axis == 0 ? 32 : 8;
    for (int comp = 0; comp < 3; ++comp) {
        const R *a = (const R *)src[comp];
        R *b = (R *)dst[comp];
        for (int c = c_first; c < 32; c += c_step) {
            const long long lo = s_line[c];
            for (int s_ = s_first; s_ < len; s_ += s_step) {
                int q = q0 + s_ - P;
                bool ok = lo >= 0;
                if (q < 0 || q >= n) {
                    // a ragged last pencil can reach more than one period past the end
                    if (per) q = ((q % n) + n) % n;
                    else ok = false;
                }
                buf[0][s_][c] = ok ? a[lo + (long long)q * sa] : R(0);
            }
        }
        __syncthreads();
        int cur = 0;
        for (int pass = 0; pass < P; ++pass) {
            for (int c = c_first; c < 32; c += c_step)
                for (int s_ = s_first; s_ < len; s_ += s_step) {
                    R v = R(0);
                    if (s_ >= 1 && s_ < len - 1) {
                        v = R(0.25) * buf[cur][s_ - 1][c] + R(0.5) * buf[cur][s_][c] + R(0.25) * buf[cur][s_ + 1][c];
                        const int q = q0 + s_ - P;
                        if (!per && (q < 0 || q >= n)) v = R(0);
                    }
                    buf[cur ^ 1][s_][c] = v;
                }
            __syncthreads();
            cur ^= 1;
        }
        for (int c = c_first; c < 32; c += c_step) {
            const long long lo = s_line[c];
            if (lo < 0) continue;
            for (int s_ = s_first; s_ < kPencil; s_ += s_step) {
                const int q = q0 + s_;
                if (q < n) b[lo + (long long)q * sa] = buf[cur][s_ + P][c];
            }
        }
        __syncthreads();
    }
}

template <typename R, int P>
__global__ void __launch_bounds__(256, sizeof(R) == 4 ? 4 : 2) k_filter_col(Launch L, int axis, const long long *pencil_start, int src_is_jt)
{
    filter_col_block<R, P>(L, axis, pencil_start, src_is_jt, blockIdx.x);
}

template <typename R, int P>
__global__ void __launch_bounds__(256) k_filter_row(Launch L, const long long *pencil_start, int src_is_jt)
{
    __shared__ R sw[8 * 3 * (kPencil + 2 * P)];
    filter_row_block<R, P>(L, pencil_start, src_is_jt, blockIdx.x, sw);
}

// Periodic ghost exchange of the six E/B components along one axis, per_inst_max
// elements per instance (ghost_elem).
template <typename R>
__global__ void __launch_bounds__(256) k_ghost(Launch L, int axis, long long per_inst_max)
{
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    const int ii = (int)(g / per_inst_max);
    if (ii >= L.ninst) return;
    const InstDev &I = L.inst[ii];
    const long long r = g - (long long)ii * per_inst_max;
    if (r < ghost_elems(I, axis)) ghost_elem<R>(I, axis, r);
}

// FP64 field energy sums (1/2) sum (E^2 + B^2) dV per instance.  Each block takes a
// contiguous range of kEnergyCells cells of the flattened cell space and, for every
// instance the range meets, sums its part (each cell's E^2 + B^2 in the storage
// precision, then FP64) and adds it with one atomic: a few thousand atomics per call on
// the same address, and blocks enough for a grid of 10^5 cells (8192 cells a block left 2M
// cells on 256 blocks: 60 us).
constexpr long long kEnergyCells = 2048;

// sum of v over the block (every thread gets it)
__device__ __forceinline__ double block_sum(double v, double *red)
{
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    __syncthreads();  // red is free
    if (lane == 0) red[warp] = v;
    __syncthreads();
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    return t;
}

template <typename R>
__global__ void __launch_bounds__(256) k_field_energy(Launch L, double *sums)
{
    __shared__ double red[8];
    const long long b0 = (long long)blockIdx.x * kEnergyCells;
    const long long b1 = min(b0 + kEnergyCells, L.total_cells);
    if (b0 >= b1) return;
    int ii = find_instance_ll(L.cell_start, L.ninst, b0);
    for (long long lo = b0; lo < b1; ++ii) {
        const long long hi = min(b1, L.cell_start[ii + 1]);
        const InstDev &I = L.inst[ii];
        const R *Ex = (const R *)eb_field(I, 0), *Ey = (const R *)eb_field(I, 1), *Ez = (const R *)eb_field(I, 2);
        const R *Bx = (const R *)eb_field(I, 3), *By = (const R *)eb_field(I, 4), *Bz = (const R *)eb_field(I, 5);
        double e = 0.0;
        for (long long g = lo + threadIdx.x; g < hi; g += blockDim.x) {
            const int r = (int)(g - L.cell_start[ii]);
            const int rq = fast_div(r, I.div_n0);
            const int i = r - rq * I.n[0];
            const int k = fast_div(rq, I.div_n1);
            const int j = rq - k * I.n[1];
            const long long p = (i + I.gh[0]) + I.sy * (j + I.gh[1]) + I.sz * (k + I.gh[2]);
            // the cell's E^2 + B^2 in the storage precision, then FP64
            R s2 = Ex[p] * Ex[p] + Bx[p] * Bx[p];
            s2 += Ey[p] * Ey[p] + By[p] * By[p];
            s2 += Ez[p] * Ez[p] + Bz[p] * Bz[p];
            e += (double)s2;
        }
        const double t = block_sum(e, red);
        if (threadIdx.x == 0 && t != 0.0) atomicAdd(sums + 2 * L.ninst + ii, t * (0.5 * I.dx[0] * I.dx[1] * I.dx[2]));
        lo = hi;
    }
}

// Interior values of one component as dense FP64 (x fastest), for the z planes k0 ..
// k0 + ncell / (n0 n1) - 1 (k0 = 0 and ncell = every cell for a whole field)
template <typename R>
__global__ void k_pack(InstDev I, int comp, int filtered, double *dense, long long ncell, int k0)
{
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= ncell) return;
    const int i = (int)(g % I.n[0]);
    const int j = (int)((g / I.n[0]) % I.n[1]);
    const int k = k0 + (int)(g / ((long long)I.n[0] * I.n[1]));
    const long long p = (i + I.gh[0]) + I.sy * (j + I.gh[1]) + I.sz * (k + I.gh[2]);
    const void *src;
    if (comp < 6) src = eb_field(I, comp);
    else {
        const int nsweeps = I.filter_passes > 0 ? (I.ndim == 3 ? 3 : 2) : 0;
        src = (filtered && (nsweeps & 1)) ? I.Jt[comp - 6] : I.J[comp - 6];
    }
    dense[g] = (double)((const R *)src)[p];
}

// The inverse of k_pack: writes (add = 0) or adds (add = 1) dense FP64 values
template <typename R>
__global__ void k_unpack(InstDev I, int comp, const double *dense, long long ncell, int k0, int add)
{
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= ncell) return;
    const int i = (int)(g % I.n[0]);
    const int j = (int)((g / I.n[0]) % I.n[1]);
    const int k = k0 + (int)(g / ((long long)I.n[0] * I.n[1]));
    const long long p = (i + I.gh[0]) + I.sy * (j + I.gh[1]) + I.sz * (k + I.gh[2]);
    R *dst = (R *)(comp < 6 ? eb_field(I, comp) : I.J[comp - 6]);
    dst[p] = add ? (R)((double)dst[p] + dense[g]) : (R)dense[g];
}

// div E on nodes: sum_a (E_a[i] - E_a[i - e_a]) / dx_a.  The quotients are divisions, not
// products with a rounded 1 / dx_a, which are up to 20 % further (rms) from the exact sum for
// spacings that are no powers of two.
template <typename R>
__global__ void k_dive(InstDev I, double *dense, long long ncell)
{
    const long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (g >= ncell) return;
    CellPos c;
    const int rq = fast_div((int)g, I.div_n0);
    c.i = (int)g - rq * I.n[0];
    c.k = fast_div(rq, I.div_n1);
    c.j = rq - c.k * I.n[1];
    c.p = (c.i + I.gh[0]) + I.sy * (c.j + I.gh[1]) + I.sz * (c.k + I.gh[2]);
    long long up[3], dn[3];
    neighbour_offsets(I, c, up, dn);
    double d = 0.0;
    for (int a = 0; a < 3; ++a) {
        if (I.ndim == 2 && a == 1) continue;
        const R *E = (const R *)eb_field(I, a);
        d += ((double)E[c.p] - (double)E[c.p + dn[a]]) / I.dx[a];
    }
    dense[g] = d;
}

// ------------------------------------------------------------------------------------
static inline unsigned blocks_for(long long n, int t) { return (unsigned)((n + t - 1) / t); }

template <typename R, int P>
static void filter_fixed(const Launch &L, int axis, unsigned nb, const long long *start, int src_is_jt, cudaStream_t s)
{
    if (axis == 0)
        k_filter_row<R, P><<<nb, 256, 0, s>>>(L, start, src_is_jt);
    else
        k_filter_col<R, P><<<nb, 256, 0, s>>>(L, axis, start, src_is_jt);
}

template <typename R>
static void filter_axis(const Launch &L, int axis, int passes, unsigned nb, const long long *start, int src_is_jt,
                        cudaStream_t s)
{
    switch (passes) {
    case 1: filter_fixed<R, 1>(L, axis, nb, start, src_is_jt, s); break;
    case 2: filter_fixed<R, 2>(L, axis, nb, start, src_is_jt, s); break;
    case 3: filter_fixed<R, 3>(L, axis, nb, start, src_is_jt, s); break;
    case 4: filter_fixed<R, 4>(L, axis, nb, start, src_is_jt, s); break;
    default: k_filter_axis<R><<<nb, 256, 0, s>>>(L, axis, start, src_is_jt); break;
    }
}

template <typename R, int ND>
static cudaError_t maxwell_fused_attr()
{
    return cudaFuncSetAttribute(k_maxwell_fused<R, ND>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)maxwell_fused_smem<R, ND, mx_warps<ND>()>());
}

template <typename R, int ND>
static void maxwell_fused_t(const Launch &L, const long long *tile_start, unsigned nb, int filtered, cudaStream_t s)
{
    k_maxwell_fused<R, ND><<<nb, 32 * mx_warps<ND>(), maxwell_fused_smem<R, ND, mx_warps<ND>()>(), s>>>(L, tile_start, filtered);
}

cudaError_t launch_maxwell_fused(int fp64, int ndim, const Launch &L, const long long *tile_start, long long ntiles,
                                 int filtered, cudaStream_t s)
{
    if (ntiles <= 0) return cudaSuccess;
    const unsigned nb = (unsigned)ntiles;
    if (fp64)
        ndim == 3 ? maxwell_fused_t<double, 3>(L, tile_start, nb, filtered, s)
                  : maxwell_fused_t<double, 2>(L, tile_start, nb, filtered, s);
    else
        ndim == 3 ? maxwell_fused_t<float, 3>(L, tile_start, nb, filtered, s)
                  : maxwell_fused_t<float, 2>(L, tile_start, nb, filtered, s);
    return cudaGetLastError();
}

cudaError_t prepare_fields(int fp64)
{
    cudaError_t e = fp64 ? maxwell_fused_attr<double, 3>() : maxwell_fused_attr<float, 3>();
    if (e == cudaSuccess) e = fp64 ? maxwell_fused_attr<double, 2>() : maxwell_fused_attr<float, 2>();
    return e;
}

cudaError_t launch_filter(int fp64, const Launch &L, const long long *const pencil_start[3],
                          const long long pencil_total[3], int ndim, int passes, cudaStream_t s)
{
    // axes in order x, (y,) z; sweep k reads J when k is even, Jt when odd
    int k = 0;
    for (int axis = 0; axis < 3; ++axis) {
        if (ndim == 2 && axis == 1) continue;
        if (pencil_total[axis] > 0) {
            const unsigned nb = (unsigned)pencil_total[axis];
            if (fp64)
                filter_axis<double>(L, axis, passes, nb, pencil_start[axis], k & 1, s);
            else
                filter_axis<float>(L, axis, passes, nb, pencil_start[axis], k & 1, s);
        }
        ++k;
    }
    return cudaGetLastError();
}

// One half step of B.  ck_n: the cells of a launch of one 3D instance under the
// low-dispersion solver, else null.  The FP32 march takes chunks of about 32 planes or, on
// smaller grids, as many as fill the 608 resident blocks once (a chunk loads two planes more
// than it puts out; 64x64x512: 8 blocks an SM 115, 4 blocks 112 us for the three updates).
// In FP64 the per-cell kernel stays: both are bound by the FP64 pipe (64x64x512: 1108 us,
// the march 1126).  2D3V and batches keep it too; no march has been written for them.
template <typename R>
static void bhalf(int solver, const Launch &L, const int *ck_n, int damp, cudaStream_t s)
{
    const unsigned nb = blocks_for(L.total_cells, 256);
    if (solver == PIC_SOLVER_CK && ck_n) {
        const long long cols = blocks_for((long long)ck_n[0] * ck_n[1], 128);
        const long long waves = (cols * ((ck_n[2] + 31) / 32) + 607) / 608;
        const int chunks = (int)std::max(1LL, std::min(608 * waves / cols, 65535LL));
        const int tz = (ck_n[2] + chunks - 1) / chunks;
        k_bhalf_ck3<<<dim3((unsigned)cols, (ck_n[2] + tz - 1) / tz), 128, 0, s>>>(L, damp, tz);
    } else if (solver == PIC_SOLVER_CK) {
        k_bhalf<R, true><<<nb, 256, 0, s>>>(L, damp);
    } else {
        k_bhalf<R, false><<<nb, 256, 0, s>>>(L, damp);
    }
}

cudaError_t launch_bhalf(int fp64, int solver, const Launch &L, const int *ck_n, int damp, cudaStream_t s)
{
    if (fp64)
        bhalf<double>(solver, L, nullptr, damp, s);
    else
        bhalf<float>(solver, L, ck_n, damp, s);
    return cudaGetLastError();
}

cudaError_t launch_maxwell(int fp64, int solver, const Launch &L, const int *ck_n, int filtered, cudaStream_t s)
{
    cudaError_t e = launch_bhalf(fp64, solver, L, ck_n, 0, s);
    if (e == cudaSuccess) e = launch_efull(fp64, L, filtered, s);
    return e == cudaSuccess ? launch_bhalf(fp64, solver, L, ck_n, 1, s) : e;
}

cudaError_t launch_efull(int fp64, const Launch &L, int filtered, cudaStream_t s)
{
    const unsigned nb = blocks_for(L.total_cells, 256);
    if (fp64)
        k_efull<double><<<nb, 256, 0, s>>>(L, filtered);
    else
        k_efull<float><<<nb, 256, 0, s>>>(L, filtered);
    return cudaGetLastError();
}

cudaError_t launch_ghost(int fp64, const Launch &L, int axis, long long per_inst_max, cudaStream_t s)
{
    const long long n = per_inst_max * L.ninst;
    if (fp64)
        k_ghost<double><<<blocks_for(n, 256), 256, 0, s>>>(L, axis, per_inst_max);
    else
        k_ghost<float><<<blocks_for(n, 256), 256, 0, s>>>(L, axis, per_inst_max);
    return cudaGetLastError();
}

cudaError_t launch_field_energy(int fp64, const Launch &L, double *sums, cudaStream_t s)
{
    const unsigned nb = (unsigned)((L.total_cells + kEnergyCells - 1) / kEnergyCells);
    if (fp64)
        k_field_energy<double><<<nb, 256, 0, s>>>(L, sums);
    else
        k_field_energy<float><<<nb, 256, 0, s>>>(L, sums);
    return cudaGetLastError();
}

cudaError_t launch_pack(int fp64, const InstDev &I, int comp, int filtered, double *dense, long long ncell, cudaStream_t s)
{
    return launch_pack_planes(fp64, I, comp, filtered, dense, 0, (int)(ncell / ((long long)I.n[0] * I.n[1])), s);
}

cudaError_t launch_unpack(int fp64, const InstDev &I, int comp, const double *dense, long long ncell, cudaStream_t s)
{
    return launch_unpack_planes(fp64, I, comp, dense, 0, (int)(ncell / ((long long)I.n[0] * I.n[1])), 0, s);
}

cudaError_t launch_pack_planes(int fp64, const InstDev &I, int comp, int filtered, double *dense, int k0, int nk,
                               cudaStream_t s)
{
    const long long n = (long long)nk * I.n[0] * I.n[1];
    if (n <= 0) return cudaSuccess;
    if (fp64) k_pack<double><<<blocks_for(n, 256), 256, 0, s>>>(I, comp, filtered, dense, n, k0);
    else k_pack<float><<<blocks_for(n, 256), 256, 0, s>>>(I, comp, filtered, dense, n, k0);
    return cudaGetLastError();
}

cudaError_t launch_unpack_planes(int fp64, const InstDev &I, int comp, const double *dense, int k0, int nk, int add,
                                 cudaStream_t s)
{
    const long long n = (long long)nk * I.n[0] * I.n[1];
    if (n <= 0) return cudaSuccess;
    if (fp64) k_unpack<double><<<blocks_for(n, 256), 256, 0, s>>>(I, comp, dense, n, k0, add);
    else k_unpack<float><<<blocks_for(n, 256), 256, 0, s>>>(I, comp, dense, n, k0, add);
    return cudaGetLastError();
}

// max |a - b| and sum (a - b)^2 over n values (FP64); the maximum is kept as the bit
// pattern of a non-negative double, which orders like the value
__global__ void __launch_bounds__(256) k_residual(const double *a, const double *b, long long n,
                                                  unsigned long long *max_bits, double *sumsq)
{
    double m = 0.0, q = 0.0;
    for (long long g = (long long)blockIdx.x * blockDim.x + threadIdx.x; g < n; g += (long long)gridDim.x * blockDim.x) {
        const double d = fabs(a[g] - b[g]);
        m = fmax(m, d);
        q += d * d;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
        m = fmax(m, __shfl_xor_sync(0xffffffffu, m, o));
        q += __shfl_xor_sync(0xffffffffu, q, o);
    }
    if ((threadIdx.x & 31) == 0) {
        atomicMax(max_bits, (unsigned long long)__double_as_longlong(m));
        atomicAdd(sumsq, q);
    }
}

cudaError_t launch_residual(const double *a, const double *b, long long n, unsigned long long *max_bits, double *sumsq,
                            cudaStream_t s)
{
    const long long blocks = std::min<long long>(blocks_for(n, 256), 152LL * 8);
    k_residual<<<(unsigned)std::max<long long>(blocks, 1), 256, 0, s>>>(a, b, n, max_bits, sumsq);
    return cudaGetLastError();
}

cudaError_t launch_dive(int fp64, const InstDev &I, double *dense, long long ncell, cudaStream_t s)
{
    if (fp64) k_dive<double><<<blocks_for(ncell, 256), 256, 0, s>>>(I, dense, ncell);
    else k_dive<float><<<blocks_for(ncell, 256), 256, 0, s>>>(I, dense, ncell);
    return cudaGetLastError();
}

}  // namespace pic
