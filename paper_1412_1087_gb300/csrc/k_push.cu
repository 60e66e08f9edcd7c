// FP64 particle step (the reference GPU path): drift, TSC gather,
// E-parallel cleaning, relativistic Boris kick-rotate-kick, drift, corrector
// deposit at x^(n+1/2) and moments deposit at x^(n+1) (App. A.1-A.3 of
// arXiv:1412.1087), the particle arithmetic in double and in the oracle's
// order but for the reciprocals.
//
// Same work decomposition as the mixed kernel (k_push_mixed.cu): persistent
// CTAs take brick items from an atomic counter, stage the brick's fields plus
// a halo in shared memory and accumulate the deposits in a shared
// fixed-point tile that is added to the global accumulators at the end; a
// particle whose stencil leaves the tile uses global memory directly.
//
// The FP64 pipe bounds it, so what need not be FP64 is not: the deposits are
// integer products (wide_fixed.cuh), gamma and 1/gamma come from one
// reciprocal square root (math64.cuh) instead of square roots and divisions,
// positions are compared and cut into cell and offset with integer
// operations (1100 -> 440 FP64 operations a particle); with the deposit tile in
// 32-bit words a step of 48^3 x 16 particles takes 2.02 ms (4.81 before).
#include "math64.cuh"
#include "push_common.cuh"
#include "wide_fixed.cuh"

namespace mhdpic {

namespace {

// Extra bits of a deposited quantity: |q| scale <= 2^62 / (9 * 64) (the
// headroom of the scales), and up to 4 times that before the overflow flag,
// so q 2^WIDE stays inside int64.
constexpr int WIDE = 8;

// The deposit tile.  W = 3: a slot is SLOT_WORDS consecutive 32-bit words, three
// for each channel: 19, 19 and the upper bits of every contribution (an item
// has at most 4,096 contributions per cell and channel, and they are below
// 2^55 or, when flagged, go to the global accumulators, so no word overflows
// before the flush puts them together); an odd slot size keeps slots that differ mod 32 on different banks.  64-bit
// shared atomic adds are compare-and-swap loops (a step of 48^3 x 16 particles
// 2.52 ms, 2.02 with three words); they remain (W = 1, a 64-bit word per
// channel) for bricks whose tile would not fit otherwise.
constexpr int SLOT_WORDS = 3 * NCH + 1;
constexpr int WORD_BITS = 19;
constexpr unsigned WORD_MASK = (1u << WORD_BITS) - 1u;

__host__ __device__ constexpr size_t f64_tile_bytes(int slots, int words)
{
    return ((words == 3 ? sizeof(unsigned) * SLOT_WORDS : sizeof(unsigned long long) * NCH) * (size_t)slots + 15) / 16 *
           16;
}

struct F64Const {
    double dt, h, C, C2, invC;
    double lo[3], L[3], hi[3];   // box bounds
    double inv_dx[3];
    double mq[4];                // -m_CR times the corrector scales
    double qn;                   // (q/mc) m / dV at the density's scale, and at the current's:
    double qj[3];
    uint64_t vlim[4];            // bits of the corrector quantities that raise the overflow flag
};

__device__ __forceinline__ void f64_const(const BoxDev &b, double dt, F64Const &k)
{
    k.dt = dt;
    k.h = b.qm_cr * dt;
    k.C = b.C;
    k.C2 = b.C * b.C;
    k.invC = 1.0 / b.C;
    for (int d = 0; d < 3; ++d) {
        k.lo[d] = b.x0[d];
        k.L[d] = b.n[d] * b.dx[d];
        k.hi[d] = k.lo[d] + k.L[d];
        k.inv_dx[d] = b.inv_dx[d];
    }
    const double qn = b.qm_cr * b.m_cr * b.inv_dV;
    k.qn = qn * b.scale[CH_N];
    for (int d = 0; d < 3; ++d)
        k.qj[d] = qn * b.scale[CH_JX + d];
    for (int ch = 0; ch < 4; ++ch) {
        k.mq[ch] = -b.m_cr * b.scale[ch];
        k.vlim[ch] = (uint64_t)__double_as_longlong(b.qmax[ch] * b.scale[ch]);
    }
}

// |q| > limit for the bits of a limit >= 0 (false for NaN)
__device__ __forceinline__ bool beyond(double q, uint64_t limit)
{
    const uint64_t a = (uint64_t)__double_as_longlong(q) & 0x7fffffffffffffffull;
    return a > limit && a <= 0x7ff0000000000000ull;
}

template <int D>
__device__ __forceinline__ void gather_f64(const Ctx &c, const BoxDev &b, bool in_tile, int base,
                                           const int ci[3], const double w[3][3], const double2 *__restrict__ sF,
                                           double E[3], double Bf[3])
{
    E[0] = E[1] = E[2] = Bf[0] = Bf[1] = Bf[2] = 0.0;
    const double2 *__restrict__ gF = reinterpret_cast<const double2 *>(c.f64);
    const int SY = c.fts[1], SZ = c.fts[2];
    int gx[3], gy[3], gz[3];
    if (!in_tile)
        stencil_coords<D>(b, ci, gx, gy, gz);
    // rolled: the code of a whole particle, unrolled, misses the instruction
    // cache (7% of the push, with the deposit a function of its own)
#pragma unroll 1
    for (int cz = 0; cz < (D == 3 ? 3 : 1); ++cz)
#pragma unroll 1
        for (int cy = 0; cy < 3; ++cy) {
            const double wyz = D == 3 ? w[1][cy] * w[2][cz] : w[1][cy];
#pragma unroll
            for (int cx = 0; cx < 3; ++cx) {
                const double ww = w[0][cx] * wyz;
                const double2 *f = sF + 3 * (base + cx + SY * cy + SZ * cz);
                if (!in_tile)
                    f = gF + 3 * (b.cell0 + ((int64_t)gz[cz] * b.n[1] + gy[cy]) * b.n[0] + gx[cx]);
                const double2 a0 = f[0], a1 = f[1], a2 = f[2];
                E[0] += ww * a0.x;
                E[1] += ww * a0.y;
                E[2] += ww * a1.x;
                Bf[0] += ww * a1.y;
                Bf[1] += ww * a2.x;
                Bf[2] += ww * a2.y;
            }
        }
}

// Cell and offset of a position.
template <int D>
__device__ __forceinline__ void cell_of_f64(const F64Const &k, const double x[3], int ci[3], double o[3])
{
#pragma unroll
    for (int d = 0; d < D; ++d)
        floor_split((x[d] - k.lo[d]) * k.inv_dx[d], ci[d], o[d]);
}

// Four channels (already at their scales) with the TSC weights of offsets o:
// into the tile when the stencil lies in it, else into the global
// accumulators; the same integers either way.
template <int D, int W>
__device__ __noinline__ void deposit4_f64(const Ctx &c, const BoxDev &b, bool in_tile, int base, const int ci[3],
                                          const double o[3], const double q[4], int ch0, void *sD,
                                          unsigned long long *__restrict__ gdst)
{
    const int S = c.tile_slots, SY = c.ts[1], SZ = c.ts[2];
    const int64_t nc = c.nc;
    uint64_t wz[3] = {0ull, 1ull << 63, 0ull}, pair[9], mag[4], sign[4];
    {
        uint64_t wx[3], wy[3];
        wide_tsc(o[0], wx);
        wide_tsc(o[1], wy);
        if (D == 3)
            wide_tsc(o[2], wz);
#pragma unroll
        for (int cy = 0; cy < 3; ++cy)
#pragma unroll
            for (int cx = 0; cx < 3; ++cx)
                pair[3 * cy + cx] = wide_pair<WIDE>(wx[cx], wy[cy]);
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
        wide_q<WIDE>(q[k], mag[k], sign[k]);
    int gx[3], gy[3], gz[3];
    if (!in_tile)
        stencil_coords<D>(b, ci, gx, gy, gz);
#pragma unroll 1
    for (int cz = 0; cz < (D == 3 ? 3 : 1); ++cz) {
        const uint64_t w = D == 3 ? (cz == 0 ? wz[0] : (cz == 1 ? wz[1] : wz[2])) : wz[1];
        uint64_t qz[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)
            qz[k] = mul_hi_round(mag[k], w);
        if (in_tile) {
#pragma unroll
            for (int n = 0; n < 9; ++n) {
                const int slot = base + n % 3 + SY * (n / 3) + SZ * cz;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                    const unsigned long long v = wide_value(qz[k], pair[n], sign[k]);
                    if (W == 3) {
                        unsigned *t = static_cast<unsigned *>(sD) + slot * SLOT_WORDS + 3 * (ch0 + k);
                        atomicAdd(t, (unsigned)v & WORD_MASK);
                        atomicAdd(t + 1, (unsigned)(v >> WORD_BITS) & WORD_MASK);
                        atomicAdd(t + 2, (unsigned)((long long)v >> (2 * WORD_BITS)));
                    } else {
                        atomicAdd(static_cast<unsigned long long *>(sD) + (ch0 + k) * S + slot, v);
                    }
                }
            }
        } else {
#pragma unroll 1
            for (int n = 0; n < 9; ++n) {
                const int64_t g = b.cell0 + ((int64_t)gz[D == 3 ? cz : 1] * b.n[1] + gy[n / 3]) * b.n[0] + gx[n % 3];
                uint64_t p = pair[0];
#pragma unroll
                for (int i = 1; i < 9; ++i)
                    p = n == i ? pair[i] : p;
#pragma unroll
                for (int k = 0; k < 4; ++k)
                    atomicAdd(gdst + k * nc + g, wide_value(qz[k], p, sign[k]));
            }
        }
    }
}

// The particle boundary along d (boundary_f64): a particle inside a periodic
// box, told by integer comparisons, only takes the rounding of x - lo + lo.
__device__ __forceinline__ bool bounded(const BoxDev &b, const F64Const &k, int d, double &x, double &vd)
{
    if (b.bc[d] == MHDPIC_BC_PERIODIC) {
        const double r = x - k.lo[d];
        if ((uint64_t)__double_as_longlong(r) < (uint64_t)__double_as_longlong(k.L[d])) {
            x = k.lo[d] + r;
            return false;
        }
    }
    return boundary_f64(b, d, x, vd);
}

template <int D, bool FULL, int W>
__device__ __forceinline__ float push_one_f64(const Ctx &c, const BoxDev &b, const ItemGeom &gm,
                                              const F64Const &k, int64_t j, const double2 *sF,
                                              void *sD, unsigned long long *mout)
{
    const int64_t np = c.np;
    const int64_t src = c.perm_src ? (int64_t)c.perm_src[j] : j;
    double x[3] = {0.0, 0.0, 0.0}, v[3];
#pragma unroll
    for (int d = 0; d < D; ++d)
        x[d] = c.src_x[d * np + src];
#pragma unroll
    for (int d = 0; d < 3; ++d)
        v[d] = c.src_p64[d * np + src];
    if (isnan(x[0])) {   // left the box earlier (kept until the next sort)
        for (int d = 0; d < D; ++d)
            c.x[d * np + j] = x[d];
        for (int d = 0; d < 3; ++d)
            c.p64[d * np + j] = 0.0;
        return 0.f;
    }

    // gamma = sqrt(C^2 + v^2)/C and its inverse from one reciprocal square
    // root; a particle at an open face is held just inside it, deposits its
    // corrector and then leaves
    const double s0 = k.C2 + (v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
    const double y0 = reciprocal_sqrt(s0);
    const double g0 = s0 * y0 * k.invC;
    bool leaving = false;
    {
        const double hu = 0.5 * k.dt * (k.C * y0);
#pragma unroll
        for (int d = 0; d < D; ++d) {
            x[d] = x[d] + hu * v[d];
            leaving |= bounded(b, k, d, x[d], v[d]);
        }
    }

    int ci[3] = {0, 0, 0}, rel[3] = {0, 0, 0};
    double o[3];
    cell_of_f64<D>(k, x, ci, o);
    bool in_tile = true;
#pragma unroll
    for (int d = 0; d < D; ++d)
        in_tile &= tile_rel(c, b, gm, d, ci[d], rel[d]);
    const int base = (rel[0] - 1) + c.ts[1] * (rel[1] - 1) + (D == 3 ? c.ts[2] * (rel[2] - 1) : 0);
    const int fbase = (rel[0] - 1) + c.fts[1] * (rel[1] - 1) + (D == 3 ? c.fts[2] * (rel[2] - 1) : 0);

    double E[3], Bf[3];
    {
        double w[3][3];
#pragma unroll
        for (int d = 0; d < D; ++d)
            tsc_from_offset<double>(o[d], w[d]);
        gather_f64<D>(c, b, in_tile, fbase, ci, w, sF, E, Bf);
    }
    const double B2 = Bf[0] * Bf[0] + Bf[1] * Bf[1] + Bf[2] * Bf[2];
    if (B2 > 0.0) {
        const double eb = (E[0] * Bf[0] + E[1] * Bf[1] + E[2] * Bf[2]) * reciprocal(B2);
#pragma unroll
        for (int d = 0; d < 3; ++d)
            E[d] -= eb * Bf[d];
    }

    const double hh = 0.5 * k.h;
    double e[3], v0[3], v1[3], vn[3], bb[3], t[3];
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        e[d] = hh * E[d];
        v0[d] = v[d] + e[d];
    }
    const double sm = k.C2 + (v0[0] * v0[0] + v0[1] * v0[1] + v0[2] * v0[2]);
    const double ym = reciprocal_sqrt(sm);
    const double gam = sm * ym * k.invC;
    const double hb = hh * (k.C * ym);
#pragma unroll
    for (int d = 0; d < 3; ++d)
        bb[d] = hb * Bf[d];
    t[0] = v0[0] + (v0[1] * bb[2] - v0[2] * bb[1]);
    t[1] = v0[1] + (v0[2] * bb[0] - v0[0] * bb[2]);
    t[2] = v0[2] + (v0[0] * bb[1] - v0[1] * bb[0]);
    const double f = 2.0 * reciprocal(1.0 + (bb[0] * bb[0] + bb[1] * bb[1] + bb[2] * bb[2]));
    v1[0] = v0[0] + f * (t[1] * bb[2] - t[2] * bb[1]);
    v1[1] = v0[1] + f * (t[2] * bb[0] - t[0] * bb[2]);
    v1[2] = v0[2] + f * (t[0] * bb[1] - t[1] * bb[0]);
#pragma unroll
    for (int d = 0; d < 3; ++d)
        vn[d] = v1[d] + e[d];

    // dE_k: the rotation keeps |v|, so the energy change is that of the two
    // half kicks, E_k(a) - E_k(b) = (a-b).(a+b)/(gamma_a+gamma_b), a-b = (h/2)E
    const double sn = k.C2 + (vn[0] * vn[0] + vn[1] * vn[1] + vn[2] * vn[2]);
    const double yn = reciprocal_sqrt(sn);
    const double g1 = sn * yn * k.invC, ig1 = k.C * yn;
    const double dEk = (e[0] * (vn[0] + v1[0]) + e[1] * (vn[1] + v1[1]) + e[2] * (vn[2] + v1[2])) * reciprocal(g1 + gam) +
                       (e[0] * (v0[0] + v[0]) + e[1] * (v0[1] + v[1]) + e[2] * (v0[2] + v[2])) * reciprocal(gam + g0);
    {
        const double qc[4] = {k.mq[0] * (vn[0] - v[0]), k.mq[1] * (vn[1] - v[1]), k.mq[2] * (vn[2] - v[2]),
                              k.mq[3] * dEk};
        const bool over = beyond(qc[0], k.vlim[0]) || beyond(qc[1], k.vlim[1]) || beyond(qc[2], k.vlim[2]) ||
                          beyond(qc[3], k.vlim[3]);
        if (over)
            set_status(c.status, MHDPIC_ST_OVERFLOW);
        deposit4_f64<D, W>(c, b, in_tile && !over, base, ci, o, qc, CH_MX, sD, c.corr);
    }

    {
        const double hu = 0.5 * k.dt * ig1;
#pragma unroll
        for (int d = 0; d < D; ++d) {
            x[d] = x[d] + hu * vn[d];
            leaving |= bounded(b, k, d, x[d], vn[d]);
        }
    }
    leaving |= removed_early(c, j);
    if (leaving) {   // removed: no moments deposit; the next sort drops it
        c.x[j] = __longlong_as_double(0x7ff8000000000000ll);
        for (int d = 1; d < D; ++d)
            c.x[d * np + j] = x[d];
        for (int d = 0; d < 3; ++d)
            c.p64[d * np + j] = 0.0;
        return 0.f;
    }
    if (FULL) {
        int rel2[3] = {0, 0, 0};
        cell_of_f64<D>(k, x, ci, o);
        bool in2 = true;
#pragma unroll
        for (int d = 0; d < D; ++d)
            in2 &= tile_rel(c, b, gm, d, ci[d], rel2[d]);
        const int base2 = (rel2[0] - 1) + c.ts[1] * (rel2[1] - 1) + (D == 3 ? c.ts[2] * (rel2[2] - 1) : 0);
        const double qm[4] = {k.qn, k.qj[0] * (vn[0] * ig1), k.qj[1] * (vn[1] * ig1), k.qj[2] * (vn[2] * ig1)};
        deposit4_f64<D, W>(c, b, in2, base2, ci, o, qm, CH_N, sD, mout);
    }
    if (!isfinite(vn[0] + vn[1] + vn[2]))
        set_status(c.status, MHDPIC_ST_NONFINITE);
#pragma unroll
    for (int d = 0; d < D; ++d)
        c.x[d * np + j] = x[d];
#pragma unroll
    for (int d = 0; d < 3; ++d)
        c.p64[d * np + j] = vn[d];
    // |v|^2 for the per-box maximum
    const float f0 = (float)vn[0], f1 = (float)vn[1], f2 = (float)vn[2];
    return f0 * f0 + f1 * f1 + f2 * f2;
}

template <int D, bool FULL, int W>
__global__ void __launch_bounds__(PUSH_THREADS, 2) k_push_f64(Ctx c, const WorkItem *__restrict__ items,
                                                          const int32_t *__restrict__ nitems,
                                                          int32_t *__restrict__ work_ctr, int cur_out,
                                                          double dt)
{
    extern __shared__ __align__(16) unsigned char smem[];
    const int S = c.tile_slots;
    int4 *clear = reinterpret_cast<int4 *>(smem);
    const unsigned *sW = reinterpret_cast<const unsigned *>(smem);
    const unsigned long long *sL = reinterpret_cast<const unsigned long long *>(smem);
    const size_t tile_bytes = f64_tile_bytes(S, W);
    double2 *sF = reinterpret_cast<double2 *>(smem + tile_bytes);
    __shared__ int s_item;
    __shared__ F64Const s_k;
    unsigned long long *mout = c.momdep[cur_out];
    const int nfront = nitems[0], nit = nfront + nitems[1];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    constexpr int NW = PUSH_THREADS / 32;

    for (;;) {
        if (threadIdx.x == 0)
            s_item = atomicAdd(work_ctr, 1);
        __syncthreads();
        const int item = s_item;
        if (item >= nit)
            break;
        const WorkItem it = work_item(c, items, nfront, item);
        const BoxDev &b = c.boxes[it.box];
        const ItemGeom gm = item_geom(c, b, it.brick, D);

        for (int s = threadIdx.x; s < (int)(tile_bytes / sizeof(int4)); s += PUSH_THREADS)
            clear[s] = make_int4(0, 0, 0, 0);
        const double2 *gF = reinterpret_cast<const double2 *>(c.f64);
        for (int t = threadIdx.x; t < c.tile_vol; t += PUSH_THREADS) {
            int tx, ty, tz;
            tile_cell(c, t, tx, ty, tz);
            int64_t g = tile_global(c, b, gm, tx, ty, tz, D);
            const int s = tx + c.fts[1] * ty + c.fts[2] * tz;
            sF[3 * s] = __ldg(gF + 3 * g);
            sF[3 * s + 1] = __ldg(gF + 3 * g + 1);
            sF[3 * s + 2] = __ldg(gF + 3 * g + 2);
        }
        if (threadIdx.x == 0)
            f64_const(b, dt, s_k);
        __syncthreads();
        const F64Const &k = s_k;

        const LaneRange lr = lane_range(it, wid, NW);
        float vm2 = 0.f;
        for (int r = lr.first; r < lr.q; r += lr.stride) {
            const int loc = lane * lr.q + r;
            if (loc < lr.cnt)
                vm2 = fmaxf(vm2, push_one_f64<D, FULL, W>(c, b, gm, k, lr.base + loc * lr.step, sF, smem, mout));
        }
        unsigned vb = __reduce_max_sync(0xffffffffu, __float_as_uint(sqrtf(vm2)));
        if (lane == 0 && vb)
            atomicMax(&c.stats[it.box].vmax, vb);
        __syncthreads();

        for (int t = threadIdx.x; t < c.tile_vol; t += PUSH_THREADS) {
            int tx, ty, tz;
            tile_cell(c, t, tx, ty, tz);
            int64_t g = tile_global(c, b, gm, tx, ty, tz, D);
            const int s = tile_slot(c, tx, ty, tz);
            for (int ch = 0; ch < (FULL ? NCH : 4); ++ch) {
                unsigned long long a;
                if (W == 3) {
                    const unsigned *t = sW + s * SLOT_WORDS + 3 * ch;
                    a = (unsigned long long)(long long)(int)t[2] << (2 * WORD_BITS);
                    a += ((unsigned long long)t[1] << WORD_BITS) + t[0];
                } else {
                    a = sL[ch * S + s];
                }
                if (a)
                    atomicAdd(ch < CH_N ? c.corr + ch * c.nc + g : mout + (ch - CH_N) * c.nc + g, a);
            }
        }
        __syncthreads();
    }
}

constexpr int PUSH_SMEM_LIMIT = 200 * 1024;

int words_f64(const Ctx &c)
{
    return f64_tile_bytes(c.tile_slots, 3) + 48 * (size_t)c.ftile_slots <= PUSH_SMEM_LIMIT ? 3 : 1;
}

// the kernel for a context's dimension and tile, with both deposits or the
// corrector's alone
auto kernel_f64(const Ctx &c, bool full)
{
    const bool w3 = words_f64(c) == 3;
    if (c.ndim == 3)
        return full ? (w3 ? k_push_f64<3, true, 3> : k_push_f64<3, true, 1>)
                    : (w3 ? k_push_f64<3, false, 3> : k_push_f64<3, false, 1>);
    return full ? (w3 ? k_push_f64<2, true, 3> : k_push_f64<2, true, 1>)
                : (w3 ? k_push_f64<2, false, 3> : k_push_f64<2, false, 1>);
}

}  // namespace

size_t push_smem_bytes_f64(const Ctx &c)
{
    return f64_tile_bytes(c.tile_slots, words_f64(c)) + 48 * (size_t)c.ftile_slots;
}

int push_blocks_per_sm_f64(const Ctx &c)
{
    int nb = 0;
    for (bool full : {false, true}) {
        auto k = kernel_f64(c, full);
        cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, PUSH_SMEM_LIMIT);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, PUSH_THREADS, push_smem_bytes_f64(c));
    }
    return nb < 1 ? 1 : nb;
}

int launch_push_f64(const Ctx &c, const SortScratch &s, int32_t *work_ctr, int cur_out, int full, double dt,
                    int grid_blocks, cudaStream_t st)
{
    cudaMemsetAsync(work_ctr, 0, sizeof(int32_t), st);
    kernel_f64(c, full != 0)<<<grid_blocks, PUSH_THREADS, push_smem_bytes_f64(c), st>>>(c, s.items, s.nitems, work_ctr,
                                                                                       cur_out, dt);
    return 1;
}

}  // namespace mhdpic
