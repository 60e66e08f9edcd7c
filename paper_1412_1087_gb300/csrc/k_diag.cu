// Diagnostics of arXiv:1412.1087: particle spectra and E_max (Section 4.3,
// eq:dpdE, eq:emax) and the CR-Hall parameter map Lambda (Section 2.2,
// eq:defR, eq:lambda).
//
// The spectrum bins a per-particle quantity (E_k = v^2/(gamma+1) or |v|)
// against caller-given edges.  What decides a bin is defined as explicitly
// rounded IEEE double operations in a fixed order (no contraction into FMAs),
// so the decision is reproducible exactly on any IEEE machine.  The FP64 pipe
// bounds the pass (a square root and two divisions are about 50 FP64
// instructions, 17 SM cycles each per warp), so the quantity is first formed
// from refined reciprocals (math64.cuh) to a few units in the last place and
// compared as integers; only one that close to a bin edge takes the defined
// operations.  In the same way the region test compares whole cells and
// forms the position only in the cells the bounds lie in or next to.  Counts
// are integers; the moment sums are reduced in a fixed order (per block of a
// fixed particle slice, then the slices), so repeated calls on the same state
// give identical results.  The energy and a region's momentum spectrum of
// 512^2 x 64 particles with the rest of an output call (the Lambda map, the
// deposit): 4.15 -> 1.79 ms.
#include <climits>

#include "device_common.cuh"
#include "math64.cuh"

namespace mhdpic {

namespace {

constexpr int SPEC_THREADS = 256;
// A quantity at most this many units in the last place from an edge is
// evaluated again in the defined operations (the fast value is within about 6).
constexpr long long NEAR_ULPS = 64;

// Doubles in their order as signed integers (NaN beyond the infinities).
__device__ __forceinline__ long long ordered(double x)
{
    const long long b = __double_as_longlong(x);
    return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}

// The binned quantity by its definition, and to a few units in the last place.
template <int KIND>
__device__ __forceinline__ double quantity_ieee(const double v[3], double C)
{
    const double v2 = __dadd_rn(__dadd_rn(__dmul_rn(v[0], v[0]), __dmul_rn(v[1], v[1])), __dmul_rn(v[2], v[2]));
    if (KIND == MHDPIC_SPEC_MOMENTUM)
        return __dsqrt_rn(v2);
    const double gam = __ddiv_rn(__dsqrt_rn(__dadd_rn(__dmul_rn(C, C), v2)), C);
    return __ddiv_rn(v2, __dadd_rn(gam, 1.0));
}

template <int KIND>
__device__ __forceinline__ double quantity_fast(const double v[3], double C2, double invC)
{
    const double v2 = fma(v[2], v[2], fma(v[1], v[1], v[0] * v[0]));
    if (KIND == MHDPIC_SPEC_MOMENTUM)
        return square_root(v2);
    return v2 * reciprocal(fma(square_root(C2 + v2), invC, 1.0));
}

// Largest bin whose lower edge is at or below q (q in [edge 0, edge nb)).
__device__ __forceinline__ int bin_of(const long long *edges, int nb, long long q)
{
    int lo = 0, hi = nb - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (edges[mid] <= q)
            lo = mid;
        else
            hi = mid - 1;
    }
    return lo;
}

// The region along one dimension in cells: a cell in [in0, in1] lies inside
// the bounds, one at or below out0 or at or above out1 outside, the others
// are decided by the position.
struct RegionCells {
    int in0, in1, out0, out1;
};

__device__ __forceinline__ RegionCells region_cells(const BoxDev &b, int d, double lo, double hi)
{
    RegionCells r;
    const double n = (double)b.n[d];
    const double far = fmax(fabs(b.x0[d]), fabs(b.x0[d] + n * b.dx[d]));
    // the rounding of a position stays well under a cell
    if (!(far * 0x1p-50 < b.dx[d])) {
        r.in0 = INT_MAX;
        r.in1 = INT_MIN;
        r.out0 = INT_MIN;
        r.out1 = INT_MAX;
        return r;
    }
    const int l = (int)floor(fmin(fmax((lo - b.x0[d]) / b.dx[d], -8.0), n + 8.0));
    const int h = (int)floor(fmin(fmax((hi - b.x0[d]) / b.dx[d], -8.0), n + 8.0));
    r.in0 = l + 2;
    r.in1 = h - 2;
    r.out0 = l - 2;
    r.out1 = h + 2;
    return r;
}

template <int PREC, int KIND>
__global__ void __launch_bounds__(SPEC_THREADS) k_spectrum_partial(Ctx c, SpecArgs a, int nchunks, int64_t per_chunk,
                                                                    unsigned long long *__restrict__ counts,
                                                                    double *__restrict__ partials)
{
    __shared__ unsigned int hist[MHDPIC_SPEC_MAX_BINS];
    __shared__ long long edges[MHDPIC_SPEC_MAX_BINS + 1];
    __shared__ double red[2][SPEC_THREADS];
    __shared__ RegionCells region[3];
    const int bx = blockIdx.y, chunk = blockIdx.x;
    const BoxDev &b = c.boxes[bx];
    const int nb = a.nbins;
    // each box takes as many of the nchunks slices as its size asks for;
    // the others add zeros
    const int nbc = box_chunks(b, per_chunk, nchunks);
    if (chunk >= nbc) {
        if (threadIdx.x < 2)
            partials[((int64_t)bx * nchunks + chunk) * 2 + threadIdx.x] = 0.0;
        return;
    }
    for (int i = threadIdx.x; i < nb; i += SPEC_THREADS)
        hist[i] = 0u;
    for (int i = threadIdx.x; i <= nb; i += SPEC_THREADS)
        edges[i] = ordered(a.edges[i]);
    if (PREC == MHDPIC_PREC_MIXED && a.has_region && threadIdx.x < c.ndim)
        region[threadIdx.x] = region_cells(b, threadIdx.x, a.region[2 * threadIdx.x], a.region[2 * threadIdx.x + 1]);
    __syncthreads();

    const double C = b.C, C2 = C * C, invC = 1.0 / C;
    const long long first = edges[0], last = edges[nb];
    long long rlo[3], rhi[3];
    for (int d = 0; d < 3; ++d) {
        rlo[d] = ordered(a.region[2 * d]);
        rhi[d] = ordered(a.region[2 * d + 1]);
    }
    const int64_t npb = b.part1 - b.part0;
    const int64_t ps = (npb + nbc - 1) / nbc;
    const int64_t p0 = b.part0 + chunk * ps, p1 = min(b.part1, p0 + ps);
    double s1 = 0.0, s0 = 0.0;
    for (int64_t i = p0 + threadIdx.x; i < p1; i += SPEC_THREADS) {
        double v[3];
        bool inside = true;
        if (PREC == MHDPIC_PREC_MIXED) {
            const int4 ps4 = c.pos[i];
            const float4 vs = c.vel[i];
            if (ps4.x == DEAD_CELL)   // left the box
                continue;
            if (a.has_region) {
                int ci[3];
                const float o[3] = {__int_as_float(ps4.y), __int_as_float(ps4.z), __int_as_float(ps4.w)};
                decode_cell(b, ps4.x, ci);
#pragma unroll
                for (int d = 0; d < 3; ++d) {
                    if (d >= c.ndim)
                        break;
                    const RegionCells r = region[d];
                    if (ci[d] <= r.out0 || ci[d] >= r.out1) {
                        inside = false;
                    } else if (ci[d] < r.in0 || ci[d] > r.in1) {
                        const double s = __dadd_rn((double)ci[d], (double)o[d]);
                        const long long xd = ordered(__dadd_rn(b.x0[d], __dmul_rn(s, b.dx[d])));
                        inside &= xd >= rlo[d] && xd < rhi[d];
                    }
                }
                if (!inside)
                    continue;
            }
#pragma unroll
            for (int d = 0; d < 3; ++d)
                v[d] = vel_f64(vs, d);   // the exact value of the two-word four-velocity
        } else {
            if (isnan(c.x[i]))   // left the box
                continue;
            if (a.has_region) {
                for (int d = 0; d < c.ndim; ++d) {
                    const double x = c.x[(int64_t)d * c.np + i];
                    inside &= x >= a.region[2 * d] && x < a.region[2 * d + 1];
                }
                if (!inside)
                    continue;
            }
#pragma unroll
            for (int d = 0; d < 3; ++d)
                v[d] = c.p64[(int64_t)d * c.np + i];
        }
        double q = quantity_fast<KIND>(v, C2, invC);
        long long key = ordered(q);
        if (!(key >= first - NEAR_ULPS && key < last + NEAR_ULPS))   // NaN as well
            continue;
        int bin = bin_of(edges, nb, key);
        if (key - edges[bin] < NEAR_ULPS || edges[bin + 1] - key <= NEAR_ULPS) {
            q = quantity_ieee<KIND>(v, C);
            key = ordered(q);
            if (!(key >= first && key < last))
                continue;
            bin = bin_of(edges, nb, key);
        }
        atomicAdd(&hist[bin], 1u);
        double qn = 1.0, pw = q;   // q^n by squaring
        for (int n = a.n_moment; n > 0; n >>= 1) {
            if (n & 1)
                qn = qn * pw;
            if (n > 1)
                pw = pw * pw;
        }
        s1 = fma(qn, q, s1);
        s0 += qn;
    }
    red[0][threadIdx.x] = s1;
    red[1][threadIdx.x] = s0;
    __syncthreads();
    for (int s = SPEC_THREADS / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
            red[0][threadIdx.x] += red[0][threadIdx.x + s];
            red[1][threadIdx.x] += red[1][threadIdx.x + s];
        }
        __syncthreads();
    }
    if (threadIdx.x < 2)
        partials[((int64_t)bx * nchunks + chunk) * 2 + threadIdx.x] = red[threadIdx.x][0];
    for (int i = threadIdx.x; i < nb; i += SPEC_THREADS)
        if (hist[i])
            atomicAdd(counts + (int64_t)bx * nb + i, (unsigned long long)hist[i]);
}

// A warp per output sums the slices (sum_slices).
__global__ void k_spectrum_final(int nbox, int nchunks, const double *__restrict__ partials,
                                 double *__restrict__ sums)
{
    const int t = (blockIdx.x * blockDim.x + threadIdx.x) >> 5;
    if (t >= nbox * 2)
        return;
    const double s = sum_slices(partials + (int64_t)(t / 2) * nchunks * 2 + t % 2, nchunks, 2);
    if ((threadIdx.x & 31) == 0)
        sums[t] = s;
}

// Lambda = (J - n v_g) / ((n_g + n) v_A) per cell, from the latest charge and
// current deposit (moments buffer cur) and the gas.  v_A = |B|/sqrt(rho) as
// |B|^2 / sqrt(|B|^2 rho); bound by the FP64 pipe.
__global__ void k_lambda(Ctx c, int cur, double *__restrict__ out)
{
    const unsigned long long *md = c.momdep[cur];
    const int64_t nc = c.nc;
    for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < nc;
         g += (int64_t)gridDim.x * blockDim.x) {
        const BoxDev &b = c.boxes[find_box(c.box_cell_start, c.nbox, g)];
        const double rho = c.rho[g];
        const double Bx = c.B[g], By = c.B[nc + g], Bz = c.B[2 * nc + g];
        const double B2 = Bx * Bx + By * By + Bz * Bz;
        const double n = from_fixed(md[g], b.inv_scale[CH_N]);
        const double ir = reciprocal(rho);
        const double vA = plain_range(B2 * rho) ? B2 * reciprocal_sqrt(B2 * rho) : sqrt(B2) / sqrt(rho);
        const double f = reciprocal((b.qm_gas * rho + n) * vA);
        for (int d = 0; d < 3; ++d) {
            const double vg = c.mom[d * nc + g] * ir;
            const double J = from_fixed(md[(1 + d) * nc + g], b.inv_scale[CH_N + 1 + d]);
            out[d * nc + g] = vA > 0.0 ? (J - n * vg) * f : 0.0;
        }
    }
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

int launch_spectrum(const Ctx &c, const SpecArgs &a, int nchunks, int64_t per_chunk, unsigned long long *counts,
                    double *partials,
                    double *sums, cudaStream_t st)
{
    cudaMemsetAsync(counts, 0, sizeof(unsigned long long) * (size_t)c.nbox * a.nbins, st);
    dim3 grid(nchunks, c.nbox);
    constexpr int M = MHDPIC_PREC_MIXED, F = MHDPIC_PREC_FP64;
    constexpr int EN = MHDPIC_SPEC_ENERGY, MO = MHDPIC_SPEC_MOMENTUM;
    auto kernel = c.prec == M ? (a.kind == EN ? k_spectrum_partial<M, EN> : k_spectrum_partial<M, MO>)
                              : (a.kind == EN ? k_spectrum_partial<F, EN> : k_spectrum_partial<F, MO>);
    kernel<<<grid, SPEC_THREADS, 0, st>>>(c, a, nchunks, per_chunk, counts, partials);
    k_spectrum_final<<<(c.nbox * 2 + 7) / 8, 256, 0, st>>>(c.nbox, nchunks, partials, sums);
    return 2;
}

int launch_lambda(const Ctx &c, int cur, double *out, cudaStream_t st)
{
    k_lambda<<<grid_for(c.nc, 256), 256, 0, st>>>(c, cur, out);
    return 1;
}

}  // namespace mhdpic
