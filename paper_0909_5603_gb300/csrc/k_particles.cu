// k_particles.cu -- particle-side helper kernels of the boosted-frame PIC step: the
// tile population scan that lays out each step's particle array, the canonical-order
// read-out, and the FP64 particle reductions and charge deposit used by the getters.
#include "k_particles.cuh"

#include <algorithm>

namespace pic {

// Source records of every tile, one warp per tile (tile_sources_warp).
__global__ void __launch_bounds__(256) k_tile_sources(Launch L)
{
    __shared__ SrcScratch W[8];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int g = blockIdx.x * 8 + warp;
    if (g >= L.total_tiles) return;  // the whole warp
    tile_sources_warp(L, g, W[warp], lane);
}

// Tile population scan, one CTA per instance (scan_instance).
__global__ void __launch_bounds__(1024) k_scan(Launch L, int mode, int *const *dst)
{
    __shared__ int sh[66];
    scan_instance(L, blockIdx.x, mode, dst, sh);
}

// -------------------------------------------------------------------------------------
// Read-out of the particles of one instance in canonical order: per destination tile, the
// same source walk as the step, into staging arrays at the scanned tile offsets.
// -------------------------------------------------------------------------------------
// read-out staging, values in the storage precision R (widened to FP64 on the host)
template <typename R>
struct Stage {
    int *cell;
    R *off;  // 3 per particle
    R *u;    // 3 per particle
    R *w;
    int *id;
};

template <typename R>
__global__ void __launch_bounds__(256) k_readout(Launch L, const int *const *start, Stage<R> out, int over)
{
    __shared__ SrcTable S;
    // the first blocks take the further windows of crowded tiles (listed by the scan)
    const InstDev &I = L.inst[0];
    const int win = readout_window(I.cap);
    int t = (int)blockIdx.x - over, part = 0;
    if (t < 0) {
        if ((int)blockIdx.x >= *I.n_over) return;
        t = I.over[blockIdx.x].x;
        part = I.over[blockIdx.x].y;
    }
    const int cur = *I.cur;
    const int tx = t % I.nt[0], ty = (t / I.nt[0]) % I.nt[1], tz = t / (I.nt[0] * I.nt[1]);
    const int dst0 = start[0][t];
    const int p0 = part * win, p1 = min(start[0][t + 1] - dst0, p0 + win);
    build_sources(I, cur, tx, ty, tz, p0, p1, S);
    for (int p = p0 + threadIdx.x; p < p1; p += blockDim.x) {
        const int pos = slot_position(I, cur, S, p);
        if (pos < 0 || pos >= I.cap) { atomicOr(I.err, kErrInternal); continue; }
        const long long q = dst0 + p;
        out.cell[q] = I.cell[cur][pos];
        out.off[3 * q + 0] = ((const R *)I.off[cur][0])[pos];
        out.off[3 * q + 1] = I.ndim == 3 ? ((const R *)I.off[cur][1])[pos] : R(0);
        out.off[3 * q + 2] = ((const R *)I.off[cur][2])[pos];
        for (int a = 0; a < 3; ++a) out.u[3 * q + a] = ((const R *)I.u[cur][a])[pos];
        out.w[q] = ((const R *)I.w[cur])[pos];
        out.id[q] = I.id[cur] ? I.id[cur][pos] : (int)q;
    }
}

// -------------------------------------------------------------------------------------
// Particle reductions of one instance for the diagnostics and the charge density: walk
// every live particle of the current layout, by chunks (their live prefix: buckets 0..26).
// Each warp of the launch takes a contiguous range of chunks, whatever tiles they belong
// to, so that a crowded tile is shared out (one block per 16 tiles left 64^3 cells with 16
// particles each on 32 blocks: 0.55 ms of a 0.77 ms diagnostics call).
// -------------------------------------------------------------------------------------
struct ChunkWalk {
    int c, end;  // chunks c .. end - 1
    int t;       // the tile of chunk c
};

__device__ __forceinline__ ChunkWalk warp_chunks(const InstDev &I, int cur)
{
    const int lane = threadIdx.x & 31;
    const int w = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), nw = gridDim.x * (blockDim.x >> 5);
    const int *base = I.chunk_base[cur];
    const int nch = base[I.ntiles];
    ChunkWalk k;
    k.c = (int)((long long)nch * w / nw);
    k.end = (int)((long long)nch * (w + 1) / nw);
    // the last tile whose chunks start at or before c: 32 probes a round
    int lo = 0;
    for (int len = I.ntiles; len > 1;) {
        const int step = (len + 31) / 32;
        const unsigned m = __ballot_sync(0xffffffffu, lane * step < len && base[lo + lane * step] <= k.c);
        const int hit = m ? 31 - __clz(m) : 0;
        lo += hit * step;
        len = min(step, len - hit * step);
    }
    k.t = lo;
    return k;
}

// Buffer position of the first particle of chunk k.c and its live particles; moves k.t on.
__device__ __forceinline__ int chunk_start(const InstDev &I, int cur, ChunkWalk &k, int &live)
{
    const int *base = I.chunk_base[cur];
    while (base[k.t + 1] <= k.c) ++k.t;
    live = I.chunk_pre[cur][(long long)k.c * kPre + kDead];
    return I.seg[cur][k.t] + (k.c - base[k.t]) * I.R;
}

// FP64 kinetic energy (without the mass) and weight sums, and the live count; one set of
// atomics per block.
template <typename R>
__global__ void __launch_bounds__(256) k_particle_sums(Launch L, double *sums, unsigned long long *n_live)
{
    __shared__ double s_ke[8], s_q[8];
    __shared__ int s_n[8];
    const InstDev &I = L.inst[0];
    const int cur = *I.cur;
    // an instance with a device error may hold a step's layout half written: its chunk
    // records are not read (the read-out reports the error instead)
    if (*(volatile const int *)I.err != 0) return;
    const R *ux = (const R *)I.u[cur][0], *uy = (const R *)I.u[cur][1], *uz = (const R *)I.u[cur][2], *wt = (const R *)I.w[cur];
    const int lane = threadIdx.x & 31;
    double ke = 0.0, q = 0.0;
    int n = 0;
    for (ChunkWalk k = warp_chunks(I, cur); k.c < k.end; ++k.c) {
        int live;
        const int start = chunk_start(I, cur, k, live);
        n += live;
#pragma unroll 8
        for (int p = lane; p < live; p += 32) {
            const int pos = start + p;  // momenta and weight only: half the particle's bytes
            const R u0 = ux[pos], u1 = uy[pos], u2 = uz[pos], w = wt[pos];
            if (sizeof(R) == 8) {
                const double g2 = 1.0 + (double)u0 * u0 + (double)u1 * u1 + (double)u2 * u2;
                ke += (double)w * (sqrt(g2) - 1.0);
            } else {
                // FP32 storage: gamma - 1 = u^2 / (1 + gamma) in FP32 (no cancellation; the
                // stored momenta carry FP32 precision anyway), summed in FP64
                const float uu = (float)u0 * (float)u0 + (float)u1 * (float)u1 + (float)u2 * (float)u2;
                ke += (double)((float)w * (uu / (1.f + sqrtf(1.f + uu))));
            }
            q += (double)w;
        }
    }
    for (int o = 16; o > 0; o >>= 1) {
        ke += __shfl_down_sync(0xffffffffu, ke, o);
        q += __shfl_down_sync(0xffffffffu, q, o);
    }
    if (lane == 0) {
        s_ke[threadIdx.x >> 5] = ke;
        s_q[threadIdx.x >> 5] = q;
        s_n[threadIdx.x >> 5] = n;
    }
    __syncthreads();
    if (threadIdx.x == 0) {
        double a = 0.0, b = 0.0;
        unsigned long long m = 0;
        for (int w = 0; w < (int)(blockDim.x >> 5); ++w) {
            a += s_ke[w];
            b += s_q[w];
            m += (unsigned long long)s_n[w];
        }
        if (m == 0) return;
        atomicAdd(sums + 0, a * I.m);
        atomicAdd(sums + 1, b * I.q);
        atomicAdd(n_live, m);
    }
}

// The diagnostics' integers beside its sums, so that one copy brings all to the host:
// sums[3] removed particles, sums[4] the error word (as 64-bit integers).
__global__ void k_diag_words(Launch L, double *sums)
{
    const InstDev &I = L.inst[0];
    unsigned long long *w = (unsigned long long *)sums;
    w[3] = *I.lost;
    w[4] = (unsigned long long)*(volatile const int *)I.err;
}

// Charge density on the nodes: per particle the wrapped node indices and the weights along
// each axis once (a weight beyond an absorbing face is zero), then products and FP64 atomics.
// The charge is divided by the cell volume per particle: with one rounded q / dV for all of
// them the density of a plasma of equal weights is off by that rounding everywhere (up to 33 %
// further from the exact sum, rms).
template <int ND, int ORD, typename R>
__global__ void __launch_bounds__(256) k_rho(Launch L, double *rho /* dense n0*n1*n2 of the instance */)
{
    const InstDev &I = L.inst[0];
    const int cur = *I.cur;
    const int *cells = I.cell[cur];
    const R *of[3] = {(const R *)I.off[cur][0], (const R *)I.off[cur][1], (const R *)I.off[cur][2]};
    const R *wt = (const R *)I.w[cur];
    const int n[3] = {I.n[0], I.n[1], I.n[2]};
    const bool per[3] = {I.bc[0] == 0, I.bc[1] == 0, I.bc[2] == 0};
    const FastDiv d0 = I.div_n0, d1 = I.div_n1;
    const double q = I.q, dV = I.dx[0] * I.dx[1] * I.dx[2];
    const int lane = threadIdx.x & 31;
    for (ChunkWalk k = warp_chunks(I, cur); k.c < k.end; ++k.c) {
        int live;
        const int start = chunk_start(I, cur, k, live);
        for (int p = lane; p < live; p += 32) {
            const int pos = start + p;
            const int c = cells[pos];
            const int cq = fast_div(c, d0);
            const int cz = ND == 3 ? fast_div(cq, d1) : cq;
            const int cc[3] = {c - cq * n[0], ND == 3 ? cq - cz * n[1] : 0, cz};
            const int st[3] = {1, n[0], n[0] * n[1]};
            double w[3][ORD + 1];
            int at[3][ORD + 1];
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                if (ND == 2 && a == 1) continue;
                const int b = shape_nodal<ORD, double>(cc[a], (double)of[a][pos], w[a]);
#pragma unroll
                for (int m = 0; m <= ORD; ++m) {
                    int x = b + m;
                    if (x < 0 || x >= n[a]) {
                        if (per[a]) x += x < 0 ? n[a] : -n[a];
                        else x = 0, w[a][m] = 0.0;
                    }
                    at[a][m] = x * st[a];
                }
            }
            const double qw = q * (double)wt[pos] / dV;
#pragma unroll
            for (int i = 0; i <= ORD; ++i) {
                const double wi = qw * w[0][i];
#pragma unroll
                for (int j = 0; j <= (ND == 3 ? ORD : 0); ++j) {
                    const double wij = ND == 3 ? wi * w[1][j] : wi;
                    double *row = rho + at[0][i] + (ND == 3 ? at[1][j] : 0);
#pragma unroll
                    for (int m = 0; m <= ORD; ++m) {
                        const double v = wij * w[2][m];
                        if (v != 0.0) atomicAdd(row + at[2][m], v);
                    }
                }
            }
        }
    }
}

// -------------------------------------------------------------------------------------
// Host-side launchers (called from pic_api.cu).
// -------------------------------------------------------------------------------------
cudaError_t dispatch_particles_f32(int ndim, int order, int pusher, const Launch *L, const OneInst *one, size_t smem,
                                   cudaStream_t s);
cudaError_t dispatch_particles_f64(int ndim, int order, int pusher, const Launch *L, const OneInst *one, size_t smem,
                                   cudaStream_t s);
cudaError_t dispatch_particles_f32_inj(int ndim, int order, int pusher, const Launch *L, const OneInst *one, size_t smem,
                                   cudaStream_t s);
cudaError_t dispatch_particles_f64_inj(int ndim, int order, int pusher, const Launch *L, const OneInst *one, size_t smem,
                                   cudaStream_t s);

static cudaError_t dispatch_particles(int ndim, int order, int fp64, int pusher, bool inj, const Launch *L,
                                      const OneInst *one, size_t smem, cudaStream_t s)
{
    if (fp64)
        return inj ? dispatch_particles_f64_inj(ndim, order, pusher, L, one, smem, s)
                   : dispatch_particles_f64(ndim, order, pusher, L, one, smem, s);
    return inj ? dispatch_particles_f32_inj(ndim, order, pusher, L, one, smem, s)
               : dispatch_particles_f32(ndim, order, pusher, L, one, smem, s);
}

cudaError_t launch_particles(int ndim, int order, int fp64, int pusher, bool inj, const Launch &L, const OneInst *one,
                             size_t smem, cudaStream_t s)
{
    return dispatch_particles(ndim, order, fp64, pusher, inj, &L, one, smem, s);
}

cudaError_t prepare_particles(int ndim, int order, int fp64, int pusher, size_t smem)
{
    cudaError_t e = dispatch_particles(ndim, order, fp64, pusher, false, nullptr, nullptr, smem, 0);
    return e == cudaSuccess ? dispatch_particles(ndim, order, fp64, pusher, true, nullptr, nullptr, smem, 0) : e;
}

int particle_chunk() { return kChunk; }
int particle_threads() { return kNT; }

cudaError_t launch_tile_sources(const Launch &L, cudaStream_t s)
{
    k_tile_sources<<<(L.total_tiles + 7) / 8, 256, 0, s>>>(L);
    return cudaGetLastError();
}

cudaError_t launch_scan(const Launch &L, int mode, int *const *dst, cudaStream_t s)
{
    k_scan<<<L.ninst, 1024, 0, s>>>(L, mode, dst);
    return cudaGetLastError();
}

cudaError_t launch_readout(int fp64, const Launch &L, int cap, const int *const *start, int *cell, void *off, void *u,
                           void *w, int *id, cudaStream_t s)
{
    const int over = cap / readout_window(cap);
    if (fp64) {
        Stage<double> st{cell, (double *)off, (double *)u, (double *)w, id};
        k_readout<double><<<L.total_tiles + over, 256, 0, s>>>(L, start, st, over);
    } else {
        Stage<float> st{cell, (float *)off, (float *)u, (float *)w, id};
        k_readout<float><<<L.total_tiles + over, 256, 0, s>>>(L, start, st, over);
    }
    return cudaGetLastError();
}

// Blocks of the chunk walks: eight for each SM, fewer when there are fewer chunks.
static unsigned walk_blocks(int chunk_cap)
{
    return (unsigned)std::max(1, std::min(152 * 8, (chunk_cap + 7) / 8));
}

cudaError_t launch_particle_sums(int fp64, const Launch &L, int chunk_cap, double *sums, cudaStream_t s)
{
    const unsigned nb = walk_blocks(chunk_cap);
    unsigned long long *n = (unsigned long long *)(sums + 5);
    if (fp64) k_particle_sums<double><<<nb, 256, 0, s>>>(L, sums, n);
    else k_particle_sums<float><<<nb, 256, 0, s>>>(L, sums, n);
    return cudaGetLastError();
}

cudaError_t launch_diag_words(const Launch &L, double *sums, cudaStream_t s)
{
    k_diag_words<<<1, 1, 0, s>>>(L, sums);
    return cudaGetLastError();
}

using RhoKernel = void (*)(Launch, double *);
static RhoKernel rho_kernel(int ndim, int order, int fp64)
{
    if (ndim == 3)
        return order == 1 ? (fp64 ? k_rho<3, 1, double> : k_rho<3, 1, float>) : (fp64 ? k_rho<3, 2, double> : k_rho<3, 2, float>);
    return order == 1 ? (fp64 ? k_rho<2, 1, double> : k_rho<2, 1, float>) : (fp64 ? k_rho<2, 2, double> : k_rho<2, 2, float>);
}

// Loads the density kernels of one (dimension, order, precision) on the current device: CUDA
// loads kernels lazily, on their first launch or attribute query.
cudaError_t preload_rho(int ndim, int order, int fp64)
{
    cudaFuncAttributes a;
    cudaError_t e = cudaFuncGetAttributes(&a, rho_kernel(ndim, order, fp64));
    return e == cudaSuccess ? preload_rho_ion() : e;
}

cudaError_t launch_rho(int order, int fp64, const Launch &L, const InstDev &I, double *rho, cudaStream_t s)
{
    rho_kernel(I.ndim, order, fp64)<<<walk_blocks(I.chunk_cap), 256, 0, s>>>(L, rho);
    cudaError_t e = cudaGetLastError();
    // plus the ion background of a lab-frame plasma
    return e == cudaSuccess && I.ion ? launch_rho_ion(L, I, rho, s) : e;
}

}  // namespace pic
