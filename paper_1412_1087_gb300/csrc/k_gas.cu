// Gas kernels of the coupled step, the predictor-corrector of App. A.3
// (eq:scheme of arXiv:1412.1087):
//
//   predictor  g^(n+1/2) = g^n + G(f^n, g^n) dt/2, with the CR sources of the
//              moments n, J deposited at x^n, fused with the staging of the
//              half-step cell fields the push reads;
//   corrector  g^(n+1) = g^n + G((f^n + f^(n+1))/2, g^(n+1/2)) dt, the CR part
//              being the corrector deposit of the push (momentum and energy
//              handed to the gas over the step).
//
// G has a CR part and a gas part.  CR sources (eq:gasmotion, eq:engeq):
// momentum -F_CR, F_CR = (1-R)(n E0 + J x B) (eq:lorentz2), energy
// -(1-R) J.E0, R = n/(n_g + n) with the CR-Hall term and 0 without it.  Gas
// part, by model:
//   MHDPIC_GAS_SOURCES   nothing else: B stays as it is;
//   MHDPIC_GAS_LINEAR_X  plane-parallel linear MHD along x (rho and B_x
//                        uniform, v_x = 0 to first order):
//                          d(rho v_y,z)/dt = B_x dB_y,z/dx,
//                          dB_y,z/dt = B_x dv_y,z/dx,
//                        plus the curl of the CR-Hall field -F_CR/n_g
//                        (eq:emfcr2 in eq:induction):
//                          dB_y/dt += -d(F_z/n_g)/dx, dB_z/dt += d(F_y/n_g)/dx;
//                        centred differences, x periodic.  In the corrector
//                        the CR-Hall field takes the force the corrector
//                        deposit implies, F_CR = -dM/(dV dt).
// The gas energy takes only the CR sources (the paper's linear test gas is
// isothermal, App. B.2).  All gas arithmetic is FP64.
#include "device_common.cuh"
#include "math64.cuh"

namespace mhdpic {

namespace {

constexpr double FIXED_LIMIT_G = 4611686018427387904.0;  // 2^62
constexpr int GAS_THREADS = 256;

__device__ __forceinline__ void cross(const double a[3], const double b[3], double o[3])
{
    o[0] = a[1] * b[2] - a[2] * b[1];
    o[1] = a[2] * b[0] - a[0] * b[2];
    o[2] = a[0] * b[1] - a[1] * b[0];
}

// Neighbour along x (s = -1 or +1) of global cell g inside box b, x periodic.
__device__ __forceinline__ int64_t x_neighbour(const BoxDev &b, int64_t g, int s)
{
    const uint32_t loc = (uint32_t)(g - b.cell0);   // a box has < 2^31 cells
    const int nx = b.n[0];
    const int i = (int)(loc - fdiv(loc, b.div_nx) * (uint32_t)nx);
    const int j = i + s < 0 ? nx - 1 : (i + s >= nx ? 0 : i + s);
    return g - i + j;
}

// n and J of the moments buffer md at cell g.
__device__ __forceinline__ void moments_at(const Ctx &c, const BoxDev &b, const unsigned long long *md, int64_t g,
                                           double &n, double J[3])
{
    const int64_t nc = c.nc;
    n = from_fixed(md[g], b.inv_scale[CH_N]);
    J[0] = from_fixed(md[nc + g], b.inv_scale[CH_JX]);
    J[1] = from_fixed(md[2 * nc + g], b.inv_scale[CH_JY]);
    J[2] = from_fixed(md[3 * nc + g], b.inv_scale[CH_JZ]);
}

// The CR sources at a cell and what the gas model takes from it: F_CR
// (eq:lorentz2), (1-R) J.E0 (eq:engeq), the gas velocity, R, and 1/rho and
// 1/n_g from refined reciprocals (FP64 divisions are slow on this GPU).
struct CellForce {
    double F[3], P, vg[3], oneR, irho, ing;
};

__device__ __forceinline__ void cr_force(const BoxDev &b, double rho, const double m[3], const double B[3], double n,
                                         const double J[3], CellForce &f)
{
    f.irho = reciprocal(rho);
    f.ing = 0.0;
    f.oneR = 1.0;
    if (b.hall) {
        const double ng = b.qm_gas * rho;
        f.ing = reciprocal(ng);
        f.oneR = 1.0 - n * reciprocal(ng + n);
    }
    for (int d = 0; d < 3; ++d)
        f.vg[d] = m[d] * f.irho;
    double vxb[3], JxB[3];
    cross(f.vg, B, vxb);
    const double E0[3] = {-vxb[0], -vxb[1], -vxb[2]};
    cross(J, B, JxB);
    for (int d = 0; d < 3; ++d)
        f.F[d] = f.oneR * (n * E0[d] + JxB[d]);
    f.P = f.oneR * (J[0] * E0[0] + J[1] * E0[1] + J[2] * E0[2]);
}

// What a cell's x neighbours need of it: the transverse gas velocity and the
// CR-Hall field F_CR / n_g.
struct Neighbour {
    double v[2], H[2];
};

__device__ __forceinline__ Neighbour neighbour_of(const CellForce &f)
{
    return {{f.vg[1], f.vg[2]}, {f.F[1] * f.ing, f.F[2] * f.ing}};
}

// The same from the state in memory (cells that another block holds).
__device__ __noinline__ Neighbour neighbour_at(const Ctx &c, const BoxDev &b, const unsigned long long *md, int64_t g)
{
    const int64_t nc = c.nc;
    double n, J[3];
    moments_at(c, b, md, g, n, J);
    const double m[3] = {c.mom[g], c.mom[nc + g], c.mom[2 * nc + g]};
    const double Bc[3] = {c.B[g], c.B[nc + g], c.B[2 * nc + g]};
    CellForce f;
    cr_force(b, c.rho[g], m, Bc, n, J, f);
    return neighbour_of(f);
}

// Predictor: half state into `half` (planes rho, mom x3, egas, B x3) and the
// cell fields of the half state (as the stage kernel: E0 = -v x B, with the
// CR-Hall term E = E0 - F/n_g from the moments at x^n) for the push; clears
// the moments buffer the next push fills; records max |E|, |B|.
//
// Bound by the FP64 pipe.  Each cell's force is formed once and its x
// neighbours read it from shared memory (forming it for both neighbours too,
// with divisions, took 190 us at 700 x 500).
template <int PREC>
__global__ void __launch_bounds__(GAS_THREADS) k_gas_predict(Ctx c, int cur, double dt, int model,
                                                            double *__restrict__ half)
{
    __shared__ Neighbour nb[GAS_THREADS];
    const unsigned long long *__restrict__ md = c.momdep[cur];
    unsigned long long *__restrict__ mnext = c.momdep[cur ^ 1];
    const int64_t nc = c.nc;
    // the loop is uniform over the block
    for (int64_t g0 = blockIdx.x * (int64_t)GAS_THREADS; g0 < nc; g0 += (int64_t)gridDim.x * GAS_THREADS) {
        const int64_t g = g0 + threadIdx.x;
        const bool in = g < nc;
        const int bx = in ? find_box(c.box_cell_start, c.nbox, g) : 0;
        const BoxDev &b = c.boxes[bx];
        double rho = 0.0, m[3], Bc[3], n = 0.0, J[3];
        CellForce f;
        if (in) {
            rho = c.rho[g];
            for (int d = 0; d < 3; ++d) {
                m[d] = c.mom[d * nc + g];
                Bc[d] = c.B[d * nc + g];
            }
            moments_at(c, b, md, g, n, J);
            cr_force(b, rho, m, Bc, n, J, f);
        }
        double dmom[3] = {0.0, 0.0, 0.0}, dB[3] = {0.0, 0.0, 0.0};
        if (model == MHDPIC_GAS_LINEAR_X) {
            __syncthreads();   // the previous cells have been read
            if (in)
                nb[threadIdx.x] = neighbour_of(f);
            __syncthreads();
            if (in) {
                const int64_t l = x_neighbour(b, g, -1), r = x_neighbour(b, g, 1);
                const bool lin = l >= g0 && l < g0 + GAS_THREADS, rin = r >= g0 && r < g0 + GAS_THREADS;
                const Neighbour L = lin ? nb[l - g0] : neighbour_at(c, b, md, l);
                const Neighbour R = rin ? nb[r - g0] : neighbour_at(c, b, md, r);
                const double h = 0.5 * b.inv_dx[0];
                for (int d = 1; d < 3; ++d) {
                    dmom[d] = Bc[0] * (c.B[d * nc + r] - c.B[d * nc + l]) * h;
                    dB[d] = Bc[0] * (R.v[d - 1] - L.v[d - 1]) * h;
                }
                if (b.hall) {
                    dB[1] -= (R.H[1] - L.H[1]) * h;
                    dB[2] += (R.H[0] - L.H[0]) * h;
                }
            }
        }
        if (!in)
            continue;
        double mh[3], Bh[3];
        for (int d = 0; d < 3; ++d) {
            mh[d] = m[d] + 0.5 * dt * (dmom[d] - f.F[d]);
            Bh[d] = Bc[d] + 0.5 * dt * dB[d];
        }
        const double egh = c.egas[g] - 0.5 * dt * f.P;
        half[g] = rho;
        half[nc + g] = mh[0];
        half[2 * nc + g] = mh[1];
        half[3 * nc + g] = mh[2];
        half[4 * nc + g] = egh;
        half[5 * nc + g] = Bh[0];
        half[6 * nc + g] = Bh[1];
        half[7 * nc + g] = Bh[2];

        // cell fields of the half state
        const double v[3] = {mh[0] * f.irho, mh[1] * f.irho, mh[2] * f.irho};
        const double E0[3] = {-(v[1] * Bh[2] - v[2] * Bh[1]), -(v[2] * Bh[0] - v[0] * Bh[2]),
                              -(v[0] * Bh[1] - v[1] * Bh[0])};
        double E[3] = {E0[0], E0[1], E0[2]};
        if (b.hall) {
            double JxB[3];
            cross(J, Bh, JxB);
            const double w = f.oneR * f.ing;
            for (int d = 0; d < 3; ++d)
                E[d] = E0[d] - w * (n * E0[d] + JxB[d]);
        }
        float em, bm;   // |E| and |B| for the per-box maxima
        if (PREC == MHDPIC_PREC_MIXED) {
            int ci[3];
            decode_cell(b, (int32_t)(g - b.cell0), ci);
            const float4 fa = make_float4((float)E[0], (float)E[1], (float)E[2], (float)Bh[0]);
            const float2 fb = make_float2((float)Bh[1], (float)Bh[2]);
            store_fields_mixed(c.fa, c.fb, b, ci[0], ci[1], ci[2], fa, fb);
            em = sqrtf(fa.x * fa.x + fa.y * fa.y + fa.z * fa.z);
            bm = sqrtf(fa.w * fa.w + fb.x * fb.x + fb.y * fb.y);
        } else {
            double2 *q = reinterpret_cast<double2 *>(c.f64) + 3 * g;
            q[0] = make_double2(E[0], E[1]);
            q[1] = make_double2(E[2], Bh[0]);
            q[2] = make_double2(Bh[1], Bh[2]);
            em = (float)sqrt(E[0] * E[0] + E[1] * E[1] + E[2] * E[2]);
            bm = (float)sqrt(Bh[0] * Bh[0] + Bh[1] * Bh[1] + Bh[2] * Bh[2]);
        }
        for (int q = 0; q < 4; ++q)
            mnext[q * nc + g] = 0ull;
        const unsigned peers = __match_any_sync(__activemask(), bx);
        const unsigned eb = __reduce_max_sync(peers, __float_as_uint(em));
        const unsigned bb = __reduce_max_sync(peers, __float_as_uint(bm));
        if ((threadIdx.x & 31) == __ffs(peers) - 1) {
            atomicMax(&c.stats[bx].emax, eb);
            atomicMax(&c.stats[bx].bmax, bb);
        }
    }
}

// Corrector: the caller's gas (c.mom, c.egas, c.B) advances from g^n to
// g^(n+1) in place; rho does not change.  Reads the half state and the
// corrector accumulators of this cell and its x neighbours; the accumulators
// are cleared by the caller after the kernel.
__global__ void k_gas_correct(Ctx c, double dt, int model, const double *__restrict__ half)
{
    const int64_t nc = c.nc;
    for (int64_t g = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; g < nc;
         g += (int64_t)gridDim.x * blockDim.x) {
        const int bx = find_box(c.box_cell_start, c.nbox, g);
        const BoxDev &b = c.boxes[bx];
        bool over = false;
        double dM[3];
        for (int d = 0; d < 3; ++d) {
            const unsigned long long a = c.corr[d * nc + g];
            over |= fabs((double)(long long)a) >= FIXED_LIMIT_G;
            dM[d] = from_fixed(a, b.inv_scale[CH_MX + d]);
        }
        const unsigned long long ae = c.corr[3 * nc + g];
        over |= fabs((double)(long long)ae) >= FIXED_LIMIT_G;
        const double dE = from_fixed(ae, b.inv_scale[CH_E]);
        double dmom[3] = {0.0, 0.0, 0.0}, dB[3] = {0.0, 0.0, 0.0};
        if (model == MHDPIC_GAS_LINEAR_X) {
            const int64_t l = x_neighbour(b, g, -1), r = x_neighbour(b, g, 1);
            const double *rho_h = half, *mom_h = half + nc, *B_h = half + 5 * nc;
            const double h = 0.5 * b.inv_dx[0], Bx = B_h[g];
            const double irl = reciprocal(rho_h[l]), irr = reciprocal(rho_h[r]);
            for (int d = 1; d < 3; ++d) {
                dmom[d] = Bx * (B_h[d * nc + r] - B_h[d * nc + l]) * h;
                dB[d] = Bx * (mom_h[d * nc + r] * irr - mom_h[d * nc + l] * irl) * h;
            }
            if (b.hall) {
                // F_CR = -dM / (dV dt), H = F_CR / n_g of the half state:
                // H = corr (-inv_scale / (dV dt qm_gas)) / rho
                const double k = -h * b.inv_dV * reciprocal(dt * b.qm_gas);
                double dH[3];
                for (int d = 1; d < 3; ++d)
                    dH[d] = (from_fixed(c.corr[d * nc + r], b.inv_scale[CH_MX + d]) * irr -
                             from_fixed(c.corr[d * nc + l], b.inv_scale[CH_MX + d]) * irl) * k;
                dB[1] -= dH[2];
                dB[2] += dH[1];
            }
        }
        for (int d = 0; d < 3; ++d) {
            c.mom[d * nc + g] += dt * dmom[d] + dM[d] * b.inv_dV;
            c.B[d * nc + g] += dt * dB[d];
        }
        c.egas[g] += dE * b.inv_dV;
        if (over)
            set_status(c.status, MHDPIC_ST_OVERFLOW);
    }
    if (blockIdx.x == 0)
        for (int q = threadIdx.x; q < c.nbox; q += blockDim.x)
            c.stats[q].corr_dirty = 0;
}

int cell_grid(int64_t nc)
{
    int64_t g = (nc + 255) / 256;
    return (int)(g < 1 ? 1 : (g > 4096 ? 4096 : g));
}

}  // namespace

int launch_gas_predict(const Ctx &c, int cur, double dt, int model, double *half, cudaStream_t st)
{
    if (c.prec == MHDPIC_PREC_MIXED)
        k_gas_predict<MHDPIC_PREC_MIXED><<<cell_grid(c.nc), 256, 0, st>>>(c, cur, dt, model, half);
    else
        k_gas_predict<MHDPIC_PREC_FP64><<<cell_grid(c.nc), 256, 0, st>>>(c, cur, dt, model, half);
    return 1;
}

int launch_gas_correct(const Ctx &c, double dt, int model, const double *half, cudaStream_t st)
{
    k_gas_correct<<<cell_grid(c.nc), 256, 0, st>>>(c, dt, model, half);
    cudaMemsetAsync(c.corr, 0, sizeof(unsigned long long) * 4 * (size_t)c.nc, st);
    return 1;
}

}  // namespace mhdpic
