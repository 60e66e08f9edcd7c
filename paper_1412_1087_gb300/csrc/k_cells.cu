// Per-cell kernels: feedback to the gas fused with the staging of the
// cell-centred fields; the standalone charge/current deposit; FP64 totals;
// read-back conversions.
#include "cells_common.cuh"
#include "math64.cuh"
#include "wide_fixed.cuh"

namespace mhdpic {

namespace {

// One pass over the cells of all boxes (prep_cells).
template <int PREC>
__global__ void k_prep(Ctx c, int cur, int apply)
{
    prep_cells<PREC>(c, cur, apply);
}

__global__ void k_scales(Ctx c, double dt)
{
    int bx = blockIdx.x * blockDim.x + threadIdx.x;
    if (bx < c.nbox)
        scales_box(c, bx, dt);
}
// FP64 precision: charge and current densities at the current positions (App.
// A.1, eq:nJCR), n = qm m W / dV, J = qm m u W / dV, straight into the global
// accumulators, a warp's particles together (group_deposit).  Bound by the
// FP64 pipe and the L2's 64-bit atomics.
constexpr int MOMENTS_SH = 8;   // |q| scale <= 2^62 / (9 * 64): q 2^8 fits int64

template <int D>
__global__ void __launch_bounds__(256) k_moments_f64(Ctx c, int cur)
{
    __shared__ WideGroup<D> groups[256 / 32];
    const int64_t np = c.np;
    for (int64_t i0 = (blockIdx.x * (int64_t)blockDim.x + threadIdx.x) & ~31ll; i0 < np;
         i0 += (int64_t)gridDim.x * blockDim.x) {
        const int64_t i = i0 + (threadIdx.x & 31);
        const bool live = i < np && !particle_dead<MHDPIC_PREC_FP64>(c, i);   // dead: left the box
        double q[4], o[3];
        int gx[3], gy[3], gz[3];
        const BoxDev &b = c.boxes[find_box(c.box_part_start, c.nbox, i < np ? i : np - 1)];
        if (live) {
            int ci[3] = {0, 0, 0};
#pragma unroll
            for (int d = 0; d < D; ++d)
                floor_split((c.x[d * np + i] - b.x0[d]) * b.inv_dx[d], ci[d], o[d]);
            double v[3];
#pragma unroll
            for (int d = 0; d < 3; ++d)
                v[d] = c.p64[d * np + i];
            const double ig = b.C * reciprocal_sqrt(b.C * b.C + (v[0] * v[0] + v[1] * v[1] + v[2] * v[2]));
            const double qn = b.qm_cr * b.m_cr * b.inv_dV;
            q[0] = qn * b.scale[CH_N];
#pragma unroll
            for (int d = 0; d < 3; ++d)
                q[1 + d] = qn * b.scale[CH_JX + d] * (v[d] * ig);
#pragma unroll
            for (int a = 0; a < 3; ++a) {
                gx[a] = map_coord(ci[0] + a - 1, b.n[0], b.bc[0]);
                gy[a] = map_coord(ci[1] + a - 1, b.n[1], b.bc[1]);
                gz[a] = D == 3 ? map_coord(ci[2] + a - 1, b.n[2], b.bc[2]) : 0;
            }
        }
        group_deposit<D, MOMENTS_SH>(groups[threadIdx.x >> 5], live, q, o, gx, gy, gz, b.cell0, b.n[0],
                                     b.n[0] * b.n[1], c.momdep[cur], 1, c.nc);
    }
}

// Deterministic FP64 totals per box: block (chunk, box) reduces a fixed slice
// of the box's cells and particles in a fixed order; a second kernel adds the
// chunks in a fixed order.  out per box: P_gas(3), E_gas, P_CR(3), E_CR.  The
// FP64 pipe bounds it: E_k from refined reciprocals (math64.cuh) instead of a
// square root and two divisions.
template <int PREC>
__global__ void __launch_bounds__(256) k_totals_partial(Ctx c, int nchunks, int64_t per_chunk, double *partials)
{
    const int bx = blockIdx.y, chunk = blockIdx.x;
    const BoxDev &b = c.boxes[bx];
    const int64_t nc = c.nc;
    // each box takes as many of the nchunks slices as its size asks for;
    // the others add zeros
    const int nbc = box_chunks(b, per_chunk, nchunks);
    if (chunk >= nbc) {
        if (threadIdx.x < 8)
            partials[((int64_t)bx * nchunks + chunk) * 8 + threadIdx.x] = 0.0;
        return;
    }
    double acc[8] = {0, 0, 0, 0, 0, 0, 0, 0};
    int64_t cs = (b.ncell + nbc - 1) / nbc;
    int64_t c0 = b.cell0 + chunk * cs, c1 = min(b.cell0 + b.ncell, c0 + cs);
    for (int64_t g = c0 + threadIdx.x; g < c1; g += blockDim.x) {
        for (int d = 0; d < 3; ++d)
            acc[d] += c.mom[d * nc + g] * b.dV;
        acc[3] += c.egas[g] * b.dV;
    }
    int64_t npb = b.part1 - b.part0;
    int64_t ps = (npb + nbc - 1) / nbc;
    int64_t p0 = b.part0 + chunk * ps, p1 = min(b.part1, p0 + ps);
    const double C2 = b.C * b.C, invC = 1.0 / b.C, m_cr = b.m_cr;
    for (int64_t i = p0 + threadIdx.x; i < p1; i += blockDim.x) {
        double v[3];
        if (PREC == MHDPIC_PREC_MIXED) {
            const float4 vs = c.vel[i];   // the exact value of the two-word four-velocity
            for (int d = 0; d < 3; ++d)
                v[d] = vel_f64(vs, d);
        } else {
            for (int d = 0; d < 3; ++d)
                v[d] = c.p64[(int64_t)d * c.np + i];
        }
        const double v2 = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
        const double s = C2 + v2;
        for (int d = 0; d < 3; ++d)
            acc[4 + d] += m_cr * v[d];
        // E_k = v^2 / (gamma + 1)
        acc[7] += m_cr * (v2 * reciprocal(fma(square_root(s), invC, 1.0)));
    }
    __shared__ double red[8][256];
    for (int q = 0; q < 8; ++q)
        red[q][threadIdx.x] = acc[q];
    __syncthreads();
    for (int s = blockDim.x / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s)
            for (int q = 0; q < 8; ++q)
                red[q][threadIdx.x] += red[q][threadIdx.x + s];
        __syncthreads();
    }
    if (threadIdx.x < 8)
        partials[((int64_t)bx * nchunks + chunk) * 8 + threadIdx.x] = red[threadIdx.x][0];
}

// A warp per box and quantity sums the slices (sum_slices).
__global__ void k_totals_final(int nbox, int nchunks, const double *partials, double *out)
{
    const int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (t >= nbox * 8)
        return;
    const double s = sum_slices(partials + (int64_t)(t / 8) * nchunks * 8 + t % 8, nchunks, 8);
    if ((threadIdx.x & 31) == 0)
        out[t] = s;
}

__global__ void k_fixed_to_double(Ctx c, const unsigned long long *__restrict__ src, int ch0,
                                  double *__restrict__ out)
{
    for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < c.nc;
         g += (int64_t)gridDim.x * blockDim.x) {
        const BoxDev &b = c.boxes[find_box(c.box_cell_start, c.nbox, g)];
        for (int q = 0; q < 4; ++q)
            out[q * c.nc + g] = from_fixed(src[q * c.nc + g], b.inv_scale[ch0 + q]);
    }
}

__global__ void k_fields_to_double(Ctx c, double *__restrict__ out)
{
    for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < c.nc;
         g += (int64_t)gridDim.x * blockDim.x) {
        if (c.prec == MHDPIC_PREC_MIXED) {
            const int bx = find_box(c.box_cell_start, c.nbox, g);
            const BoxDev &b = c.boxes[bx];
            int ci[3];
            decode_cell(b, (int32_t)(g - b.cell0), ci);
            const int64_t f = fidx(b, ci[0], ci[1], ci[2]);
            const float4 a = c.fa[f];
            const float2 bb = c.fb[f];
            const float v[6] = {a.x, a.y, a.z, a.w, bb.x, bb.y};
            for (int q = 0; q < 6; ++q)
                out[q * c.nc + g] = (double)v[q];
        } else {
            for (int q = 0; q < 6; ++q)
                out[q * c.nc + g] = c.f64[g * 6 + q];
        }
    }
}

// The current four-velocities as double, plane-major: the exact value of each
// two-word record in mixed precision, a copy in FP64.
__global__ void k_velocities_to_double(Ctx c, double *__restrict__ out)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < c.np;
         i += (int64_t)gridDim.x * blockDim.x) {
        if (c.prec == MHDPIC_PREC_MIXED) {
            const float4 vs = c.vel[i];
            for (int d = 0; d < 3; ++d)
                out[d * c.np + i] = vel_f64(vs, d);
        } else {
            for (int d = 0; d < 3; ++d)
                out[d * c.np + i] = c.p64[d * c.np + i];
        }
    }
}

// FP64 precision: largest |v| per box (for the fixed-point scales; in mixed
// precision the deposit records it): a running maximum per
// thread while its particles stay in one box, one atomic per box and warp.
__global__ void k_vmax(Ctx c)
{
    float acc = 0.f;
    int bacc = -1;
    auto flush = [&](int bx, float vm) {
        const unsigned active = __activemask();
        const unsigned peers = __match_any_sync(active, bx);
        const unsigned m = __reduce_max_sync(peers, __float_as_uint(vm));
        if (bx >= 0 && m && (threadIdx.x & 31) == __ffs(peers) - 1)
            atomicMax(&c.stats[bx].vmax, m);
    };
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < c.np;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int bx = find_box(c.box_part_start, c.nbox, i);
        double v2 = 0.0;
        for (int d = 0; d < 3; ++d) {
            const double v = c.p64[(int64_t)d * c.np + i];
            v2 += v * v;
        }
        float vm = (float)sqrt(v2);
        if (!(vm <= 1.0e37f))
            vm = 1.0e37f;
        if (bx != bacc) {   // rare: a thread's particles cross into the next box
            if (bacc >= 0 && acc > 0.f)
                atomicMax(&c.stats[bacc].vmax, __float_as_uint(acc));
            bacc = bx;
            acc = 0.f;
        }
        acc = fmaxf(acc, vm);
    }
    flush(bacc, acc);
}

int grid_for(int64_t n, int threads)
{
    int64_t b = (n + threads - 1) / threads;
    if (b < 1)
        b = 1;
    if (b > 152 * 32)
        b = 152 * 32;
    return (int)b;
}

}  // namespace

int launch_prep(const Ctx &c, int cur, int apply, cudaStream_t st)
{
    // small boxes: a block for every 32 cells (see prep_cells)
    const int64_t groups = (c.nc + 31) / 32;
    const int grid = groups <= 152 * 8 ? (int)(groups < 1 ? 1 : groups) : grid_for(c.nc, 256);
    if (c.prec == MHDPIC_PREC_MIXED)
        k_prep<MHDPIC_PREC_MIXED><<<grid, 256, 0, st>>>(c, cur, apply);
    else
        k_prep<MHDPIC_PREC_FP64><<<grid, 256, 0, st>>>(c, cur, apply);
    return 1;
}

int launch_moments(const Ctx &c, int cur, cudaStream_t st)
{
    cudaMemsetAsync(c.momdep[cur], 0, sizeof(unsigned long long) * 4 * c.nc, st);
    if (c.np == 0)
        return 0;
    const int g = grid_for(c.np, 256);
    if (c.ndim == 3)
        k_moments_f64<3><<<g, 256, 0, st>>>(c, cur);
    else
        k_moments_f64<2><<<g, 256, 0, st>>>(c, cur);
    return 1;
}

int launch_totals(const Ctx &c, double *partials, int nchunks, int64_t per_chunk, double *out, cudaStream_t st)
{
    dim3 grid(nchunks, c.nbox);
    if (c.prec == MHDPIC_PREC_MIXED)
        k_totals_partial<MHDPIC_PREC_MIXED><<<grid, 256, 0, st>>>(c, nchunks, per_chunk, partials);
    else
        k_totals_partial<MHDPIC_PREC_FP64><<<grid, 256, 0, st>>>(c, nchunks, per_chunk, partials);
    k_totals_final<<<c.nbox, 256, 0, st>>>(c.nbox, nchunks, partials, out);
    return 2;
}

int launch_fixed_to_double(const Ctx &c, const unsigned long long *src, int ch0, double *out,
                           cudaStream_t st)
{
    k_fixed_to_double<<<grid_for(c.nc, 256), 256, 0, st>>>(c, src, ch0, out);
    return 1;
}

int launch_fields_to_double(const Ctx &c, double *out, cudaStream_t st)
{
    k_fields_to_double<<<grid_for(c.nc, 256), 256, 0, st>>>(c, out);
    return 1;
}

int launch_velocities_to_double(const Ctx &c, double *out, cudaStream_t st)
{
    if (c.np == 0)
        return 0;
    k_velocities_to_double<<<grid_for(c.np, 256), 256, 0, st>>>(c, out);
    return 1;
}

int launch_vmax(const Ctx &c, cudaStream_t st)
{
    if (c.np == 0)
        return 0;
    k_vmax<<<grid_for(c.np, 256), 256, 0, st>>>(c);
    return 1;
}

int launch_scales(const Ctx &c, double dt, cudaStream_t st)
{
    k_scales<<<(c.nbox + 127) / 128, 128, 0, st>>>(c, dt);
    return 1;
}

}  // namespace mhdpic
