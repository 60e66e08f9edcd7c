// Cell sort of the particles (the library's layout; the paper has no sort).
//
// Stable counting sort by key = brick number * brick volume + cell number in
// the brick (x fastest at both levels), per box, keys of later boxes after
// earlier ones.  Steps:
//   1. key of each particle, rank among equal keys by warp-aggregated atomics
//      (this rank is not yet the stable one);
//   2. exclusive scan of the per-key counts (one kernel up to 8 tiles of 4096
//      keys, two beyond);
//   3. scatter of the particle indices to their key segment and, in the same
//      launch, the push work list;
//   4. sort of each key segment by particle index, which makes the result the
//      stable order: the permutation equals a stable sort by key.
// The particle arrays are permuted later: by the next push, which reads its
// particles through the permutation, or by launch_gather.
// The work list cuts every brick's particle range into items of at most
// item_cap particles.  At 64^2 x 16 particles a sort is launches and latency:
// 12 kernels and 5 memsets took 60 us, 5 kernels and one memset take 25.
#include <climits>

#include "async_copy.cuh"
#include "device_common.cuh"
#include "math64.cuh"

namespace mhdpic {

namespace {

constexpr int SCAN_THREADS = 1024;
constexpr int SCAN_PER_THREAD = 4;
constexpr int SCAN_TILE = SCAN_THREADS * SCAN_PER_THREAD;
constexpr int WARP_SORT_MAX = 1024;     // per-warp shared-memory bitonic sort
constexpr int BLOCK_SORT_MAX = 8192;    // per-block shared-memory bitonic sort
constexpr int RANK_SORT_MAX = 1 << 20;  // quadratic ranking beyond that is refused

__device__ __forceinline__ int64_t brick_key(const BoxDev &b, const Ctx &c, int ci, int cj, int ck)
{
    int q[3], r[3];
    const int cc[3] = {ci, cj, ck};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        if (c.brick_sh[d] >= 0) {   // power-of-two bricks: shifts and masks
            q[d] = cc[d] >> c.brick_sh[d];
            r[d] = cc[d] & (c.brick[d] - 1);
        } else {
            q[d] = cc[d] / c.brick[d];
            r[d] = cc[d] - q[d] * c.brick[d];
        }
    }
    const int64_t bid = ((int64_t)q[2] * b.nb[1] + q[1]) * b.nb[0] + q[0];
    const int64_t in = ((int64_t)r[2] * c.brick[1] + r[1]) * c.brick[0] + r[0];
    return b.key0 + bid * ((int64_t)c.brick[0] * c.brick[1] * c.brick[2]) + in;
}

// Cells a particle moves along each of the first D dimensions in time t at
// its current four-velocity v (the sort's look-ahead), -1, 0 or +1: whether
// the position o + (t/dx) v/gamma leaves its cell through the lower or the
// upper face (a half step moves a particle well under one cell).  With the
// box's FP32 constants k = {t/dx, t/dy, t/dz, 1/C^2} (each rounded once, on
// the host), g2 = gamma^2 = 1 + v^2 k.w and a_d = k_d, the faces are tested on
// squares, so that no square root or division is needed:
//   +1 when v_d > 0 and (a_d v_d)^2 >= ((1 - o_d)(1 - o_d)) g2,
//   -1 when v_d < 0 and (a_d v_d)^2 >  (o_d o_d) g2,
// v^2 = (vx vx + vy vy) + vz vz, every operation a correctly rounded FP32 one
// in this order (no contraction), so the key can be recomputed exactly
// elsewhere.
__device__ __forceinline__ void ahead_cells(const float4 k, const float v[3], const float o[3], int D, int cells[3])
{
    const float v2 = __fadd_rn(__fadd_rn(__fmul_rn(v[0], v[0]), __fmul_rn(v[1], v[1])), __fmul_rn(v[2], v[2]));
    const float g2 = __fadd_rn(1.f, __fmul_rn(v2, k.w));
    const float ta[3] = {k.x, k.y, k.z};
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        if (d >= D)
            break;
        const float av = __fmul_rn(ta[d], v[d]);
        const float l = __fmul_rn(av, av);
        const float up = __fsub_rn(1.f, o[d]);
        const float ru = __fmul_rn(__fmul_rn(up, up), g2);
        const float rl = __fmul_rn(__fmul_rn(o[d], o[d]), g2);
        cells[d] = (v[d] > 0.f && l >= ru) ? 1 : ((v[d] < 0.f && l > rl) ? -1 : 0);
    }
}

// Clamp or wrap a key cell into the box, and its brick-major key.
__device__ __forceinline__ int32_t key_of_cell(const Ctx &c, const BoxDev &b, int ci[3], bool ahead)
{
    if (ahead)
        for (int d = 0; d < c.ndim; ++d)
            ci[d] = b.bc[d] == MHDPIC_BC_PERIODIC ? map_coord(ci[d], b.n[d], MHDPIC_BC_PERIODIC)
                                                  : (ci[d] < 0 ? 0 : (ci[d] >= b.n[d] ? b.n[d] - 1 : ci[d]));
    for (int d = 0; d < 3; ++d)   // defensive: a key outside the box would index out of range
        ci[d] = ci[d] < 0 ? 0 : (ci[d] >= b.n[d] ? b.n[d] - 1 : ci[d]);
    return (int32_t)brick_key(b, c, ci[0], ci[1], ci[2]);
}

// What the mixed-precision key needs of a box, held in registers while a
// thread's particles stay in one box (reloaded when the box changes).
struct KeyBox {
    int box;
    int n[3], bc[3], nb[3];
    int32_t ncell;
    int32_t key0;   // keys are int32: the box's first key
    FastDiv dnx, dnxy;
    float4 sk;
};

__device__ __forceinline__ void load_keybox(const Ctx &c, int bx, KeyBox &kb)
{
    const BoxDev &b = c.boxes[bx];
    kb.box = bx;
#pragma unroll
    for (int d = 0; d < 3; ++d) {
        kb.n[d] = b.n[d];
        kb.bc[d] = b.bc[d];
        kb.nb[d] = b.nb[d];
    }
    kb.ncell = (int32_t)b.ncell;
    kb.key0 = (int32_t)b.key0;
    kb.dnx = b.div_nx;
    kb.dnxy = b.div_nxy;
    kb.sk = __ldg(c.sort_k + bx);
}

// Mixed precision: the key of a particle from its two records (loaded by
// the caller, so that the loads of several particles are in flight at once),
// as key_of_cell / brick_key compute it.
template <int D, bool AHEAD>
__device__ __forceinline__ int32_t key_mixed(const Ctx &c, const KeyBox &kb, const int4 ps, const float4 vs)
{
    int32_t cl = ps.x;
    if (cl == DEAD_CELL)   // particles that left the box share one key after all the others
        return (int32_t)c.nkeys;
    if (cl < 0 || cl >= kb.ncell) {
        set_status(c.status, MHDPIC_ST_CELL_RANGE);
        cl = cl < 0 ? 0 : kb.ncell - 1;
    }
    const uint32_t uc = (uint32_t)cl;
    const uint32_t kz = fdiv(uc, kb.dnxy);
    const uint32_t rr = uc - kz * kb.dnxy.d;
    const uint32_t jy = fdiv(rr, kb.dnx);
    int ci[3] = {(int)(rr - jy * kb.dnx.d), (int)jy, (int)kz};
    if (AHEAD) {
        const float v[3] = {vs.x, vs.y, vs.z};
        const float o[3] = {__int_as_float(ps.y), __int_as_float(ps.z), __int_as_float(ps.w)};
        int k[3] = {0, 0, 0};
        ahead_cells(kb.sk, v, o, D, k);
#pragma unroll
        for (int d = 0; d < D; ++d) {
            const int g = ci[d] + k[d];
            ci[d] = kb.bc[d] == MHDPIC_BC_PERIODIC ? (g < 0 ? g + kb.n[d] : (g >= kb.n[d] ? g - kb.n[d] : g))
                                                   : (g < 0 ? 0 : (g >= kb.n[d] ? kb.n[d] - 1 : g));
        }
    }
    int q[3] = {0, 0, 0}, r[3] = {0, 0, 0};
#pragma unroll
    for (int d = 0; d < D; ++d) {
        if (c.brick_sh[d] >= 0) {
            q[d] = ci[d] >> c.brick_sh[d];
            r[d] = ci[d] & (c.brick[d] - 1);
        } else {
            q[d] = ci[d] / c.brick[d];
            r[d] = ci[d] - q[d] * c.brick[d];
        }
    }
    // int32 throughout: every key of the context is below nkeys < 2^31
    const int bid = (q[2] * kb.nb[1] + q[1]) * kb.nb[0] + q[0];
    const int in = (r[2] * c.brick[1] + r[1]) * c.brick[0] + r[0];
    return kb.key0 + bid * (c.brick[0] * c.brick[1] * c.brick[2]) + in;
}

// FP64 precision: the key of particle i of box b, from its absolute position.
__device__ __forceinline__ int32_t key_f64(const Ctx &c, const BoxDev &b, int bx, int64_t i)
{
    int ci[3] = {0, 0, 0};
    const bool ahead = c.sort_ahead != 0.0;
    double x[3];
    for (int d = 0; d < c.ndim; ++d)
        x[d] = c.x[(int64_t)d * c.np + i];
    if (isnan(x[0]))   // particles that left the box share one key after all the others
        return (int32_t)c.nkeys;
    float o[3] = {0.f, 0.f, 0.f};
    for (int d = 0; d < c.ndim; ++d) {
        // dividing by a power of two is multiplying by its inverse, exactly
        // (the FP64 pipe bounds this pass: 210 us at 48^3 x 16 with divisions
        // and conversions to and from integers)
        const bool pow2 = (__double_as_longlong(b.dx[d]) & 0xfffffffffffffll) == 0;
        const double s = pow2 ? (x[d] - b.x0[d]) * b.inv_dx[d] : (x[d] - b.x0[d]) / b.dx[d];
        if (s >= 0.0 && s < (double)b.n[d]) {
            double rest;
            floor_split(s, ci[d], rest);
            o[d] = (float)rest;
        } else {
            set_status(c.status, MHDPIC_ST_CELL_RANGE);
            ci[d] = s >= (double)b.n[d] ? b.n[d] - 1 : 0;
            o[d] = (float)(s - (double)ci[d]);
        }
    }
    if (ahead) {
        const float v[3] = {(float)c.p64[i], (float)c.p64[c.np + i], (float)c.p64[2 * c.np + i]};
        int k[3] = {0, 0, 0};
        ahead_cells(__ldg(c.sort_k + bx), v, o, c.ndim, k);
        for (int d = 0; d < c.ndim; ++d)
            ci[d] += k[d];
    }
    return key_of_cell(c, b, ci, ahead);
}

// Particles handled per thread and loop pass by the streaming sort kernels:
// independent loads (and atomics) in flight hide their latency.
constexpr int SORT_ILP = 4;

// Runs of equal keys in consecutive lanes (the input is nearly sorted) take
// one atomic per run, made by the run's first lane; the rank inside the run
// is the lane offset.  Lanes outside `active` take no part; a negative key
// takes no atomic.
struct RunSlot {
    int start;   // first lane of the run
    int base;    // first slot of the run (at the first lane)
};

__device__ __forceinline__ RunSlot run_reserve(int32_t key, int lane, unsigned active, int32_t *count)
{
    const int prev = __shfl_up_sync(active, key, 1);
    const bool head = lane == 0 || !((active >> (lane - 1)) & 1u) || prev != key;
    const unsigned heads = __ballot_sync(active, head);
    RunSlot r;
    r.start = 31 - __clz(heads & (0xffffffffu >> (31 - lane)));    // last head at or below lane
    const unsigned after = heads & ~(0xffffffffu >> (31 - lane));  // heads above lane
    const int end = after ? __ffs(after) - 1 : 32;
    const unsigned tail = (end < 32 ? (1u << end) : 0u) - 1u;      // lanes below end
    const int len = __popc(active & tail & ~((1u << r.start) - 1u));
    r.base = 0;
    if (head && key >= 0)
        r.base = atomicAdd(count + key, len);
    return r;
}

__device__ __forceinline__ int32_t run_slot(const RunSlot &r, int lane, unsigned active)
{
    return __shfl_sync(active, r.base, r.start) + (lane - r.start);
}

// FP64 precision: the keys from the absolute positions, SORT_ILP particles
// per thread and pass.
__global__ void k_sort_keys_f64(Ctx c, int32_t *__restrict__ count, int32_t *__restrict__ pkey,
                                int32_t *__restrict__ pslot)
{
    const int lane = threadIdx.x & 31;
    const int64_t stride = (int64_t)gridDim.x * blockDim.x;
    for (int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i0 < c.np; i0 += SORT_ILP * stride) {
        // lanes past the end take keys no other lane has, so they form runs
        // of their own and take no atomic
        const unsigned active = __activemask();
        int32_t key[SORT_ILP];
#pragma unroll
        for (int u = 0; u < SORT_ILP; ++u) {
            const int64_t i = i0 + u * stride;
            int bx = 0;
            if (i < c.np)
                bx = find_box(c.box_part_start, c.nbox, i);
            key[u] = i < c.np ? key_f64(c, c.boxes[bx], bx, i) : -1 - lane;
        }
        RunSlot rs[SORT_ILP];
#pragma unroll
        for (int u = 0; u < SORT_ILP; ++u)
            rs[u] = run_reserve(key[u], lane, active, count);
#pragma unroll
        for (int u = 0; u < SORT_ILP; ++u) {
            const int32_t slot = run_slot(rs[u], lane, active);
            const int64_t i = i0 + u * stride;
            if (i < c.np) {
                pkey[i] = key[u];
                pslot[i] = slot;
            }
        }
    }
}

// Mixed precision, records staged: the particle records stream through a
// ring of KEY_STAGES shared-memory stages of KEY_CHUNK particles, each filled
// by one bulk copy per record array that the block's first thread issues
// KEY_STAGES chunks ahead, so the loads of later chunks are in flight while
// the keys and the atomics of this one are done.  (Two stages, 32 KB, let 5
// blocks share an SM; 3 and 4 stages measured slower at 128^3 x 32.)  A block takes the chunks
// blockIdx.x, blockIdx.x + gridDim.x, ...; each warp's 32 lanes take 32
// consecutive particles, as the run detection needs.
constexpr int KEY_THREADS = 256;
constexpr int KEY_PER_THREAD = 2;
constexpr int KEY_CHUNK = KEY_THREADS * KEY_PER_THREAD;
constexpr int KEY_STAGES = 2;
constexpr size_t KEY_SMEM = (size_t)KEY_STAGES * KEY_CHUNK * (sizeof(int4) + sizeof(float4));

// Thread 0: the copies of chunk `chunk` into one stage (the velocities only
// when the key looks ahead).
__device__ __forceinline__ void issue_records(const Ctx &c, int64_t chunk, int4 *dp, float4 *dv, bool ahead,
                                              uint64_t *bar)
{
    const int64_t p0 = chunk * KEY_CHUNK;
    const int64_t left = c.np - p0;
    const unsigned bytes = (unsigned)(left < KEY_CHUNK ? left : KEY_CHUNK) * 16u;
    mbar_expect_tx(bar, ahead ? 2u * bytes : bytes);
    bulk_copy(dp, c.pos + p0, bytes, bar);
    if (ahead)
        bulk_copy(dv, c.vel + p0, bytes, bar);
}

template <int D, bool AHEAD>
__global__ void __launch_bounds__(KEY_THREADS) k_sort_keys_staged(Ctx c, int32_t *__restrict__ count,
                                                                  int32_t *__restrict__ pkey,
                                                                  int32_t *__restrict__ pslot)
{
    extern __shared__ __align__(128) unsigned char smem[];
    int4 *sp = reinterpret_cast<int4 *>(smem);
    float4 *sv = reinterpret_cast<float4 *>(smem + (size_t)KEY_STAGES * KEY_CHUNK * sizeof(int4));
    __shared__ __align__(8) uint64_t full[KEY_STAGES];
    const int lane = threadIdx.x & 31;
    constexpr bool ahead = AHEAD;
    const int64_t nchunk = (c.np + KEY_CHUNK - 1) / KEY_CHUNK;
    const int64_t mine = (int64_t)blockIdx.x < nchunk ? (nchunk - 1 - blockIdx.x) / gridDim.x + 1 : 0;
    if (threadIdx.x == 0) {
        for (int st = 0; st < KEY_STAGES; ++st)
            mbar_init(&full[st]);
        fence_proxy_async();
        for (int64_t k = 0; k < KEY_STAGES && k < mine; ++k)
            issue_records(c, blockIdx.x + k * gridDim.x, sp + k * KEY_CHUNK, sv + k * KEY_CHUNK, ahead, &full[k]);
    }
    __syncthreads();
    KeyBox kb;
    load_keybox(c, 0, kb);
    for (int64_t k = 0; k < mine; ++k) {
        const int st = (int)(k % KEY_STAGES);
        const bool ok = mbar_wait(&full[st], (unsigned)((k / KEY_STAGES) & 1), c.copy_limit_ns);
        if (__syncthreads_or(!ok)) {
            // give up the launch, after the copies in flight have had their time
            if (threadIdx.x == 0) {
                set_status(c.status, MHDPIC_ST_COPY_TIMEOUT);
                for (int64_t j = k; j < mine && j < k + KEY_STAGES; ++j)
                    mbar_wait(&full[j % KEY_STAGES], (unsigned)((j / KEY_STAGES) & 1), COPY_LIMIT_NS);
            }
            return;
        }
        const int64_t p0 = (blockIdx.x + k * gridDim.x) * (int64_t)KEY_CHUNK;
        const int n = (int)(c.np - p0 < KEY_CHUNK ? c.np - p0 : KEY_CHUNK);
        int cbox = 0;   // the chunk's box, or -1 when it spans several
        if (c.nbox > 1) {
            const int b0 = find_box(c.box_part_start, c.nbox, p0);
            cbox = b0 == find_box(c.box_part_start, c.nbox, p0 + n - 1) ? b0 : -1;
        }
        int32_t key[KEY_PER_THREAD];
#pragma unroll
        for (int u = 0; u < KEY_PER_THREAD; ++u) {
            const int p = u * KEY_THREADS + threadIdx.x;
            key[u] = -1 - lane;   // past the end: a run of its own, no atomic
            if (p < n) {
                const int bx = cbox >= 0 ? cbox : find_box(c.box_part_start, c.nbox, p0 + p);
                if (bx != kb.box)
                    load_keybox(c, bx, kb);
                const float4 vs = ahead ? sv[st * KEY_CHUNK + p] : make_float4(0.f, 0.f, 0.f, 0.f);
                key[u] = key_mixed<D, AHEAD>(c, kb, sp[st * KEY_CHUNK + p], vs);
            }
        }
        RunSlot rs[KEY_PER_THREAD];
#pragma unroll
        for (int u = 0; u < KEY_PER_THREAD; ++u)
            rs[u] = run_reserve(key[u], lane, 0xffffffffu, count);
#pragma unroll
        for (int u = 0; u < KEY_PER_THREAD; ++u) {
            const int32_t slot = run_slot(rs[u], lane, 0xffffffffu);
            const int p = u * KEY_THREADS + threadIdx.x;
            if (p < n) {
                pkey[p0 + p] = key[u];
                pslot[p0 + p] = slot;
            }
        }
        __syncthreads();   // every thread has read the stage
        if (threadIdx.x == 0 && k + KEY_STAGES < mine) {
            fence_proxy_async();
            issue_records(c, blockIdx.x + (k + KEY_STAGES) * gridDim.x, sp + st * KEY_CHUNK, sv + st * KEY_CHUNK,
                          ahead, &full[st]);
        }
    }
}

// --- exclusive scan of int32 (values and totals < 2^31) ---

__device__ __forceinline__ int block_exclusive_scan(int v, int *warp_sums, int *total)
{
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int x = v;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o)
            x += y;
    }
    if (lane == 31)
        warp_sums[wid] = x;
    __syncthreads();
    if (wid == 0) {
        int nw = blockDim.x >> 5;
        int s = lane < nw ? warp_sums[lane] : 0;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            int y = __shfl_up_sync(0xffffffffu, s, o);
            if (lane >= o)
                s += y;
        }
        if (lane < nw)
            warp_sums[lane] = s;
    }
    __syncthreads();
    int pre = (wid > 0 ? warp_sums[wid - 1] : 0) + x - v;
    if (total)
        *total = warp_sums[(blockDim.x >> 5) - 1];
    __syncthreads();
    return pre;
}

// The thread's SCAN_PER_THREAD counts of one tile (zeros past the end).
__device__ __forceinline__ int4 scan_load(const int32_t *__restrict__ in, int64_t base, int64_t n)
{
    static_assert(SCAN_PER_THREAD == 4, "one 16-byte load per thread");
    if (base + 3 < n)
        return __ldg(reinterpret_cast<const int4 *>(in + base));
    int4 v = make_int4(0, 0, 0, 0);
    if (base < n)
        v.x = in[base];
    if (base + 1 < n)
        v.y = in[base + 1];
    if (base + 2 < n)
        v.z = in[base + 2];
    return v;
}

__global__ void k_scan_tiles(const int32_t *__restrict__ in, int64_t n, int32_t *__restrict__ sums)
{
    __shared__ int ws[32];
    const int4 v = scan_load(in, blockIdx.x * (int64_t)SCAN_TILE + (int64_t)threadIdx.x * SCAN_PER_THREAD, n);
    int tot;
    block_exclusive_scan(v.x + v.y + v.z + v.w, ws, &tot);
    if (threadIdx.x == 0)
        sums[blockIdx.x] = tot;
}

// Exclusive scan of tile blockIdx.x.  What lies before it is the sum of the
// tiles before, from `sums` or, with sums null, added up from the counts.
__global__ void k_scan_apply(const int32_t *__restrict__ in, int64_t n,
                             const int32_t *__restrict__ sums, int32_t *__restrict__ out)
{
    __shared__ int ws[32];
    int before = 0;
    if (sums) {
        for (int t = threadIdx.x; t < (int)blockIdx.x; t += SCAN_THREADS)
            before += sums[t];
    } else {
        for (int t = 0; t < (int)blockIdx.x; ++t) {
            const int4 v = scan_load(in, t * (int64_t)SCAN_TILE + (int64_t)threadIdx.x * SCAN_PER_THREAD, n);
            before += v.x + v.y + v.z + v.w;
        }
    }
    int carry;
    block_exclusive_scan(before, ws, &carry);
    const int64_t base = blockIdx.x * (int64_t)SCAN_TILE + (int64_t)threadIdx.x * SCAN_PER_THREAD;
    const int4 v = scan_load(in, base, n);
    int pre = block_exclusive_scan(v.x + v.y + v.z + v.w, ws, nullptr) + carry;
    const int vals[SCAN_PER_THREAD] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int k = 0; k < SCAN_PER_THREAD; ++k) {
        if (base + k < n)
            out[base + k] = pre;
        pre += vals[k];
    }
    // the thread holding the last element closes the array with the total
    if (base <= n - 1 && n - 1 < base + SCAN_PER_THREAD)
        out[n] = pre;
}

// out[0..n] = exclusive scan of in[0..n), out[n] = total (n >= 1).  Up to
// SCAN_DIRECT tiles each block adds up the counts of the tiles before its own
// (one launch instead of three); beyond, a first launch sums the tiles and
// each block adds up the sums before it, at 2 million keys 512 of them (at
// most one load per thread up to 4 million keys, a few dozen at 134 million:
// too little for a launch of its own).
constexpr int SCAN_DIRECT = 8;

int scan(const int32_t *in, int64_t n, int32_t *out, int32_t *tmp, cudaStream_t st)
{
    const int nt = (int)((n + SCAN_TILE - 1) / SCAN_TILE);
    if (nt <= SCAN_DIRECT) {
        k_scan_apply<<<nt, SCAN_THREADS, 0, st>>>(in, n, nullptr, out);
        return 1;
    }
    k_scan_tiles<<<nt, SCAN_THREADS, 0, st>>>(in, n, tmp);
    k_scan_apply<<<nt, SCAN_THREADS, 0, st>>>(in, n, tmp, out);
    return 2;
}

// Items of a brick of cnt particles, na of them in its first half.
__device__ __forceinline__ int brick_items(const Ctx &c, int cnt, int na)
{
    if (cnt <= c.item_cap)
        return cnt > 0 ? 1 : 0;
    if (!c.halves)
        return (cnt + c.item_cap - 1) / c.item_cap;
    return (na + c.item_cap - 1) / c.item_cap + (cnt - na + c.item_cap - 1) / c.item_cap;
}

// The push work list, SORT_THREADS consecutive bricks per block and pass:
// their items go to a range of the list that the block reserves (the order of
// the ranges does not matter: the deposits are integer sums).  Bricks of less
// than item_big particles (the ragged edge of a box, sparse regions) go to the
// far end of the array, backwards, and are pushed last (work_item), where they
// fill the blocks that run out first.
constexpr int SORT_THREADS = 256;

__device__ __forceinline__ void write_items(const Ctx &c, const int64_t *__restrict__ brick_start,
                                            const int32_t *__restrict__ offset, WorkItem *__restrict__ items,
                                            int32_t *__restrict__ nitems, int block, int nblocks)
{
    __shared__ int ws[32];
    __shared__ int s_first[2];
    const int vol = c.brick[0] * c.brick[1] * c.brick[2];
    for (int64_t g0 = (int64_t)block * SORT_THREADS; g0 < c.nbricks_total; g0 += (int64_t)nblocks * SORT_THREADS) {
        const int64_t gb = g0 + threadIdx.x;
        WorkItem w;
        int64_t pm = 0;
        int m = 0;
        if (gb < c.nbricks_total) {
            w.box = find_box(brick_start, c.nbox, gb);
            const BoxDev &b = c.boxes[w.box];
            w.brick = (int32_t)(gb - b.brick0);
            const int64_t k0 = b.key0 + (int64_t)w.brick * vol;
            w.p0 = offset[k0];
            w.p1 = offset[k0 + vol];
            pm = c.halves ? (int64_t)offset[k0 + vol / 2] : w.p1;
            m = brick_items(c, (int)(w.p1 - w.p0), (int)(pm - w.p0));
        }
        const bool small = m > 0 && w.p1 - w.p0 < c.item_big;
        int tot, small_tot;
        const int pre = block_exclusive_scan(small ? 0 : m, ws, &tot);
        const int small_pre = block_exclusive_scan(small ? m : 0, ws, &small_tot);
        if (threadIdx.x == 0) {
            s_first[0] = tot > 0 ? atomicAdd(nitems, tot) : 0;
            s_first[1] = small_tot > 0 ? atomicAdd(nitems + 1, small_tot) : 0;
        }
        __syncthreads();
        int64_t o = small ? c.items_size - 1 - (s_first[1] + small_pre) : s_first[0] + pre;
        if (m > 0 && w.p1 - w.p0 <= c.item_cap) {
            // one item; a whole 64-cell brick splits at its 32nd cell (the
            // start of the second half)
            w.pm = c.halves ? pm : -1;
            w.step = 1;
            w.count = (int32_t)(w.p1 - w.p0);
            items[o] = w;
        } else if (m > 0) {
            // crowded: each part (the two halves, or the whole brick) into
            // m_p interleaved items, item t taking positions t, t + m_p, ...
            const int64_t lo[2] = {w.p0, pm}, hi[2] = {pm, w.p1};
            for (int part = 0; part < 2; ++part) {
                const int64_t n = hi[part] - lo[part];
                const int mp = (int)((n + c.item_cap - 1) / c.item_cap);
                for (int t = 0; t < mp; ++t) {
                    w.p0 = lo[part] + t;
                    w.p1 = hi[part];
                    w.pm = -1;
                    w.step = mp;
                    w.count = (int32_t)((n - t + mp - 1) / mp);
                    items[o++] = w;
                }
            }
        }
        __syncthreads();   // s_first and ws are free again
    }
}

// Scatter (blocks below scatter_blocks) and the push work list (the blocks
// after them); both need only the offsets.  A key outside [0, nkeys] (only
// after a key pass that gave up part of its work) is flagged and its particle
// skipped.
__global__ void __launch_bounds__(SORT_THREADS) k_sort_scatter(Ctx c, const int64_t *__restrict__ brick_start,
                                                               const int32_t *__restrict__ pkey,
                                                               const int32_t *__restrict__ pslot,
                                                               const int32_t *__restrict__ offset,
                                                               int32_t *__restrict__ perm,
                                                               WorkItem *__restrict__ items,
                                                               int32_t *__restrict__ nitems, int scatter_blocks)
{
    if ((int)blockIdx.x >= scatter_blocks) {
        write_items(c, brick_start, offset, items, nitems, blockIdx.x - scatter_blocks, gridDim.x - scatter_blocks);
        return;
    }
    const int64_t np = c.np, nkeys = c.nkeys;
    uint32_t *status = c.status;
    const int64_t stride = (int64_t)scatter_blocks * blockDim.x;
    for (int64_t i0 = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i0 < np; i0 += SORT_ILP * stride) {
        int32_t key[SORT_ILP], slot[SORT_ILP];
#pragma unroll
        for (int u = 0; u < SORT_ILP; ++u) {
            const int64_t i = i0 + u * stride;
            key[u] = i < np ? pkey[i] : 0;
            slot[u] = i < np ? pslot[i] : 0;
            if (key[u] < 0 || key[u] > nkeys) {
                set_status(status, MHDPIC_ST_SORT_CAP);
                key[u] = 0;
                slot[u] = -1 - (int32_t)np;   // lands outside [0, np): not written
            }
        }
        int32_t off[SORT_ILP];
#pragma unroll
        for (int u = 0; u < SORT_ILP; ++u)
            off[u] = i0 + u * stride < np ? offset[key[u]] : 0;
#pragma unroll
        for (int u = 0; u < SORT_ILP; ++u) {
            const int64_t i = i0 + u * stride;
            if (i >= np)
                continue;
            const int64_t dst = (int64_t)off[u] + slot[u];
            if (dst >= 0 && dst < np)
                perm[dst] = (int32_t)i;
            else
                set_status(status, MHDPIC_ST_SORT_CAP);
        }
    }
}

// Ascending bitonic sort of the 32 E values a[e*32 + lane] = v[e] held by a
// warp: distances below 32 exchange through shuffles, larger ones between a
// lane's own registers.
template <int E>
__device__ __forceinline__ void warp_bitonic(int (&v)[E], int lane)
{
#pragma unroll
    for (int k = 2; k <= 32 * E; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (j >= 32) {
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const int pe = e ^ (j >> 5);
                    if (pe > e) {
                        const bool up = ((e * 32 + lane) & k) == 0;
                        const int x = v[e], y = v[pe];
                        if ((x > y) == up) {
                            v[e] = y;
                            v[pe] = x;
                        }
                    }
                }
            } else {
#pragma unroll
                for (int e = 0; e < E; ++e) {
                    const int o = __shfl_xor_sync(0xffffffffu, v[e], j);
                    const bool up = ((e * 32 + lane) & k) == 0;
                    const bool lower = (lane & j) == 0;
                    v[e] = (lower == up) ? min(v[e], o) : max(v[e], o);
                }
            }
        }
    }
}

// Sort of one segment [s, s + n), n <= 32 E, in registers, read from src
// (perm + s itself, or a copy of it); a segment already in ascending order is
// left alone.
template <int E>
__device__ __forceinline__ void warp_sort_segment(const int32_t *src, int32_t *__restrict__ perm, int s, int n,
                                                  int lane)
{
    int v[E];
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int i = e * 32 + lane;
        v[e] = i < n ? src[i] : INT_MAX;
    }
    bool ok = true;
#pragma unroll
    for (int e = 0; e < E; ++e) {
        int nxt = __shfl_down_sync(0xffffffffu, v[e], 1);
        if (e + 1 < E) {
            const int first = __shfl_sync(0xffffffffu, v[e + 1 < E ? e + 1 : e], 0);
            if (lane == 31)
                nxt = first;
        }
        const int i = e * 32 + lane;
        ok &= i >= n - 1 || v[e] < nxt;
    }
    if (__all_sync(0xffffffffu, ok))
        return;
    warp_bitonic<E>(v, lane);
#pragma unroll
    for (int e = 0; e < E; ++e) {
        const int i = e * 32 + lane;
        if (i < n)
            perm[s + i] = v[e];
    }
}

// A segment of the scatter is made of runs: each warp of the key pass gives
// the lanes of a run of equal keys consecutive slots, so a run is an
// increasing interval of consecutive particle indices, and runs never
// overlap.  Sorting such a segment only sorts its runs by their first index.
constexpr int MERGE_RUNS = 128;   // runs a warp merges (4 per lane)

// Ascending bitonic sort of the 128 values v[e] (element e*32 + lane) of a warp.
__device__ __forceinline__ void warp_bitonic64(long long (&v)[4], int lane)
{
#pragma unroll
    for (int k = 2; k <= 128; k <<= 1) {
#pragma unroll
        for (int j = k >> 1; j > 0; j >>= 1) {
            if (j >= 32) {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const int pe = e ^ (j >> 5);
                    if (pe > e) {
                        const bool up = ((e * 32 + lane) & k) == 0;
                        const long long x = v[e], y = v[pe];
                        if ((x > y) == up) {
                            v[e] = y;
                            v[pe] = x;
                        }
                    }
                }
            } else {
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const long long o = __shfl_xor_sync(0xffffffffu, v[e], j);
                    const bool up = ((e * 32 + lane) & k) == 0;
                    const bool lower = (lane & j) == 0;
                    v[e] = (lower == up) ? min(v[e], o) : max(v[e], o);
                }
            }
        }
    }
}

// Segment a[0, n) in the warp's shared memory, at most MERGE_RUNS runs: the
// sorted order into perm[s, s + n).  Returns false (nothing written) with more.
__device__ __forceinline__ bool warp_merge_runs(const int32_t *a, int n, int32_t *__restrict__ perm, int s,
                                                int lane, int *hpos)
{
    int nruns = 0;
    for (int base = 0; base < n; base += 32) {
        const int i = base + lane;
        const bool head = i < n && (i == 0 || a[i] != a[i - 1] + 1);
        const unsigned m = __ballot_sync(0xffffffffu, head);
        if (head) {
            const int pos = nruns + __popc(m & ((1u << lane) - 1u));
            if (pos < MERGE_RUNS)
                hpos[pos] = i;
        }
        nruns += __popc(m);
    }
    __syncwarp();
    if (nruns > MERGE_RUNS)
        return false;
    // (first index, run number) of each run, sorted across the warp
    long long v[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int r = e * 32 + lane;
        v[e] = r < nruns ? ((long long)a[hpos[r]] << 8) | r : LLONG_MAX;
    }
    warp_bitonic64(v, lane);
    int carry = 0;   // elements of the sorted runs before this group of 32
#pragma unroll
    for (int e = 0; e < 4; ++e) {
        const int rr = e * 32 + lane;
        int st = 0, len = 0;
        if (rr < nruns) {
            const int r = (int)(v[e] & 0xff);
            st = hpos[r];
            len = (r + 1 < nruns ? hpos[r + 1] : n) - st;
        }
        int incl = len;   // inclusive scan of the lengths in sorted order
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o)
                incl += y;
        }
        const int dst = carry + incl - len;
        for (int q = 0; q < len; ++q)
            perm[s + dst + q] = a[st + q];
        carry += __shfl_sync(0xffffffffu, incl, 31);
    }
    __syncwarp();
    return true;
}

// One segment [s, s + n) of 128 < n <= WARP_SORT_MAX by a warp, through its
// shared-memory buffer: by its runs when they are at most MERGE_RUNS, else by
// a bitonic network.
__device__ __forceinline__ void sort_mid_segment(int s, int n, int32_t *__restrict__ perm, int32_t *a, int *hp,
                                                 int lane)
{
    int P = 64;
    while (P < n)
        P <<= 1;
    for (int i = lane; i < P; i += 32)
        a[i] = i < n ? perm[s + i] : INT_MAX;
    __syncwarp();
    if (warp_merge_runs(a, n, perm, s, lane, hp))
        return;
    for (int kk = 2; kk <= P; kk <<= 1) {
        for (int j = kk >> 1; j > 0; j >>= 1) {
            for (int i = lane; i < P; i += 32) {
                int ixj = i ^ j;
                if (ixj > i) {
                    int x = a[i], y = a[ixj];
                    bool asc = (i & kk) == 0;
                    if ((x > y) == asc) {
                        a[i] = y;
                        a[ixj] = x;
                    }
                }
            }
            __syncwarp();
        }
    }
    for (int i = lane; i < n; i += 32)
        perm[s + i] = a[i];
    __syncwarp();
}

// A warp takes `group` consecutive keys (at most SEG_GROUP) at a time: their
// offsets in one load (one per lane), and, when the group's particles fit the
// warp's buffer, all of them in one coalesced pass, so that the loads of a
// whole group are in flight together; each segment of up to 128 is then sorted
// in registers.  Longer segments are listed for k_sort_long (crowded cells lie
// side by side: sorted here, one warp would take all of a group's in turn):
// up to WARP_SORT_MAX from the front of the list, the others from its end.
constexpr int SEG_GROUP = 31;
// Particles of a warp's buffer.  Its size lets 5 blocks of 8 warps share an SM,
// not 6: 6 make the SM keep 228 KB as shared memory instead of 196, it stays so
// when a push of another context starts on it (which needs less), and that
// push has half the L1 for its particle records (3% of the 128^3 x 32 step
// with three contexts at work; a stated split on every launch costs 1% where
// one is).  k_sort_long likewise.
constexpr int SEG_BUFFER = 1200;

__device__ __forceinline__ void sort_short_segment(const int32_t *src, int32_t *__restrict__ perm, int s, int n,
                                                   int lane)
{
    if (n <= 1)
        return;
    if (n <= 32)
        warp_sort_segment<1>(src, perm, s, n, lane);
    else if (n <= 64)
        warp_sort_segment<2>(src, perm, s, n, lane);
    else
        warp_sort_segment<4>(src, perm, s, n, lane);
}

__global__ void __launch_bounds__(256) k_sort_segments(int64_t nkeys, int group, const int32_t *__restrict__ offset,
                                                       int32_t *__restrict__ perm,
                                                       int32_t *__restrict__ long_list,
                                                       int32_t *__restrict__ long_count)
{
    __shared__ int32_t buf[8][SEG_BUFFER];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    int32_t *a = buf[wid];
    const int64_t nwarps = (int64_t)gridDim.x * (blockDim.x >> 5);
    for (int64_t k0 = ((int64_t)blockIdx.x * (blockDim.x >> 5) + wid) * group; k0 < nkeys;
         k0 += nwarps * group) {
        const int nk = (int)(nkeys - k0 < group ? nkeys - k0 : group);
        const int o = lane <= nk ? offset[k0 + lane] : 0;   // offsets of keys k0 .. k0 + nk
        const int gs = __shfl_sync(0xffffffffu, o, 0), ge = __shfl_sync(0xffffffffu, o, nk);
        const int len = __shfl_down_sync(0xffffffffu, o, 1) - o;
        // the long segments of the group go to the list
        const bool mid = lane < nk && len > 128 && len <= WARP_SORT_MAX, big = lane < nk && len > WARP_SORT_MAX;
        const unsigned mids = __ballot_sync(0xffffffffu, mid), bigs = __ballot_sync(0xffffffffu, big);
        if (mids | bigs) {
            int at = 0;
            if (lane == 0 && mids)
                at = atomicAdd(long_count, __popc(mids));
            if (lane == 1 && bigs)
                at = atomicAdd(long_count + 1, __popc(bigs));
            const int m0 = __shfl_sync(0xffffffffu, at, 0), b0 = __shfl_sync(0xffffffffu, at, 1);
            const unsigned below = (1u << lane) - 1u;
            if (mid)
                long_list[m0 + __popc(mids & below)] = (int32_t)(k0 + lane);
            if (big)
                long_list[nkeys - (b0 + __popc(bigs & below))] = (int32_t)(k0 + lane);
        }
        unsigned todo = __ballot_sync(0xffffffffu, lane < nk && len > 1 && len <= 128);
        const bool staged = ge - gs <= SEG_BUFFER;
        if (staged && todo) {
            for (int i = lane; i < ge - gs; i += 32)
                a[i] = perm[gs + i];
            __syncwarp();
        }
        for (; todo; todo &= todo - 1u) {
            const int j = __ffs(todo) - 1;
            const int s = __shfl_sync(0xffffffffu, o, j), n = __shfl_sync(0xffffffffu, len, j);
            sort_short_segment(staged ? a + (s - gs) : perm + s, perm, s, n, lane);
        }
        __syncwarp();   // the buffer is free again
    }
}

// The listed segments: a warp each up to WARP_SORT_MAX (the buffers of the
// block's 8 warps), then a block each: bitonic sort in shared memory up to
// BLOCK_SORT_MAX, or a quadratic ranking (elements are distinct particle
// indices) through `scratch` beyond that.
__global__ void __launch_bounds__(256) k_sort_long(int64_t nkeys, const int32_t *__restrict__ offset,
                                                   int32_t *__restrict__ perm,
                                                   const int32_t *__restrict__ long_list,
                                                   const int32_t *__restrict__ long_count,
                                                   int32_t *__restrict__ scratch, uint32_t *status)
{
    static_assert(BLOCK_SORT_MAX == 8 * WARP_SORT_MAX && SEG_BUFFER - WARP_SORT_MAX >= MERGE_RUNS,
                  "one buffer, by warps or whole, and the warps' run lists after it");
    __shared__ int32_t a[8 * SEG_BUFFER];
    int *const hp = a + BLOCK_SORT_MAX + (threadIdx.x >> 5) * MERGE_RUNS;
    const int nm = long_count[0], nb = long_count[1];
    const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
    for (int q = blockIdx.x * 8 + wid; q < nm; q += gridDim.x * 8) {
        const int64_t k = long_list[q];
        const int s = offset[k];
        sort_mid_segment(s, offset[k + 1] - s, perm, a + wid * WARP_SORT_MAX, hp, lane);
    }
    __syncthreads();   // the warps' buffers are free
    for (int q = blockIdx.x; q < nb; q += gridDim.x) {
        const int64_t k = long_list[nkeys - q];
        int s = offset[k], e = offset[k + 1];
        int n = e - s;
        if (n <= BLOCK_SORT_MAX) {
            int P = 64;
            while (P < n)
                P <<= 1;
            for (int i = threadIdx.x; i < P; i += blockDim.x)
                a[i] = i < n ? perm[s + i] : INT_MAX;
            __syncthreads();
            for (int kk = 2; kk <= P; kk <<= 1) {
                for (int j = kk >> 1; j > 0; j >>= 1) {
                    for (int i = threadIdx.x; i < P; i += blockDim.x) {
                        int ixj = i ^ j;
                        if (ixj > i) {
                            int x = a[i], y = a[ixj];
                            bool asc = (i & kk) == 0;
                            if ((x > y) == asc) {
                                a[i] = y;
                                a[ixj] = x;
                            }
                        }
                    }
                    __syncthreads();
                }
            }
            for (int i = threadIdx.x; i < n; i += blockDim.x)
                perm[s + i] = a[i];
            __syncthreads();
        } else if (n <= RANK_SORT_MAX) {
            for (int i = threadIdx.x; i < n; i += blockDim.x) {
                int v = perm[s + i];
                int r = 0;
                for (int j = 0; j < n; ++j)
                    r += perm[s + j] < v;
                scratch[s + r] = v;
            }
            __syncthreads();
            for (int i = threadIdx.x; i < n; i += blockDim.x)
                perm[s + i] = scratch[s + i];
            __syncthreads();
        } else if (threadIdx.x == 0) {
            set_status(status, MHDPIC_ST_SORT_CAP);
        }
    }
}

// All particle arrays gathered through the permutation in one pass: every
// plane q of element size esz[q] (4 or 8 bytes) is read at perm[r] and written
// at r.
struct Planes {
    const void *src[8];
    void *dst[8];
    int esz[8];
    int n;
};

__global__ void k_gather_all(int64_t np, const int32_t *__restrict__ perm, Planes pl)
{
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < np;
         r += (int64_t)gridDim.x * blockDim.x) {
        int64_t i = perm[r];
        if (i < 0 || i >= np)   // never taken for a valid permutation
            i = r;
        for (int q = 0; q < pl.n; ++q) {
            if (pl.esz[q] == 16)
                reinterpret_cast<int4 *>(pl.dst[q])[r] = __ldg(reinterpret_cast<const int4 *>(pl.src[q]) + i);
            else if (pl.esz[q] == 8)
                reinterpret_cast<unsigned long long *>(pl.dst[q])[r] =
                    __ldg(reinterpret_cast<const unsigned long long *>(pl.src[q]) + i);
            else
                reinterpret_cast<unsigned int *>(pl.dst[q])[r] =
                    __ldg(reinterpret_cast<const unsigned int *>(pl.src[q]) + i);
        }
    }
}

__global__ void k_perm_out(int64_t np, const int32_t *__restrict__ perm, int64_t *__restrict__ out)
{
    for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < np;
         r += (int64_t)gridDim.x * blockDim.x)
        out[r] = perm[r];
}

__global__ void k_max_count(int64_t n, const int32_t *__restrict__ count, int32_t *out)
{
    int m = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < n;
         i += (int64_t)gridDim.x * blockDim.x)
        m = max(m, count[i]);
    for (int o = 16; o > 0; o >>= 1)
        m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    if ((threadIdx.x & 31) == 0)
        atomicMax(out, m);
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

// Persistent grid of the staged key pass: as many blocks as fit on the
// device at once, at most one per chunk.
int key_grid(int64_t np)
{
    static int resident = 0;   // blocks of k_sort_keys_staged the device holds at once
    if (resident == 0) {
        int dev = 0, nsm = 0, per = 0;
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
        cudaFuncSetAttribute(k_sort_keys_staged<3, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)KEY_SMEM);
        cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, k_sort_keys_staged<3, true>, KEY_THREADS, KEY_SMEM);
        resident = (per < 1 ? 1 : per) * (nsm < 1 ? 1 : nsm);
    }
    const int64_t chunks = (np + KEY_CHUNK - 1) / KEY_CHUNK;
    return (int)(chunks < resident ? (chunks < 1 ? 1 : chunks) : resident);
}

template <int D, bool AHEAD>
void launch_keys(const Ctx &c, const SortScratch &s, cudaStream_t st)
{
    cudaFuncSetAttribute(k_sort_keys_staged<D, AHEAD>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)KEY_SMEM);
    k_sort_keys_staged<D, AHEAD><<<key_grid(c.np), KEY_THREADS, KEY_SMEM, st>>>(c, s.count, s.pkey, s.pslot);
}

}  // namespace

int launch_sort(const Ctx &c, const SortScratch &s, int64_t *perm_out, int32_t *counts_out,
                cudaStream_t st)
{
    int launches = 0;
    // the counts and, after them, the counters of this sort
    cudaMemsetAsync(s.count, 0, sizeof(int32_t) * (c.nkeys + 2 + SORT_COUNTERS), st);
    if (c.np > 0) {
        if (c.prec == MHDPIC_PREC_MIXED) {
            const bool ahead = c.sort_ahead != 0.0;
            if (c.ndim == 3 && ahead)
                launch_keys<3, true>(c, s, st);
            else if (c.ndim == 3)
                launch_keys<3, false>(c, s, st);
            else if (ahead)
                launch_keys<2, true>(c, s, st);
            else
                launch_keys<2, false>(c, s, st);
        } else
            k_sort_keys_f64<<<grid_for(c.np, 256), 256, 0, st>>>(c, s.count, s.pkey, s.pslot);
        ++launches;
    }
    // key nkeys holds the particles that left the box: offset[nkeys] is the
    // number of live particles
    launches += scan(s.count, c.nkeys + 1, s.offset, s.scan_tmp, st);
    const int sb = c.np > 0 ? grid_for(c.np, SORT_THREADS) : 0;
    k_sort_scatter<<<sb + grid_for(c.nbricks_total, SORT_THREADS), SORT_THREADS, 0, st>>>(
        c, s.brick_start, s.pkey, s.pslot, s.offset, s.perm, s.items, s.nitems, sb);
    ++launches;
    if (c.np > 0) {
        // as many keys per warp as keep every resident warp at work (5 blocks
        // of 8 warps per SM), at most SEG_GROUP: at 4,096 keys one each, 4 us
        // against 18 with 31
        const int64_t fit = (c.nkeys + 152 * 40 - 1) / (152 * 40);
        const int group = (int)(fit < SEG_GROUP ? (fit < 1 ? 1 : fit) : SEG_GROUP);
        const int64_t nw = (c.nkeys + 8 * group - 1) / (8 * group);   // blocks of 8 warps
        int gb = (int)(nw < 152 * 16 ? (nw < 1 ? 1 : nw) : 152 * 16);
        k_sort_segments<<<gb, 256, 0, st>>>(c.nkeys, group, s.offset, s.perm, s.long_list, s.long_count);
        // no more warps than segments of over 128 there can be
        const int64_t lw = (c.np / 128 + 7) / 8;
        k_sort_long<<<(int)(lw < 1 ? 1 : (lw < 152 * 5 ? lw : 152 * 5)), 256, 0, st>>>(
            c.nkeys, s.offset, s.perm, s.long_list, s.long_count, s.pkey, c.status);
        launches += 2;
        if (perm_out) {
            k_perm_out<<<grid_for(c.np, 256), 256, 0, st>>>(c.np, s.perm, perm_out);
            ++launches;
        }
    }
    if (counts_out)
        cudaMemcpyAsync(counts_out, s.count, sizeof(int32_t) * c.nkeys, cudaMemcpyDeviceToDevice, st);
    return launches;
}

int launch_gather(const Ctx &c, const int32_t *perm, const PSet &src, const PSet &dst, cudaStream_t st)
{
    if (c.np <= 0)
        return 0;
    Planes pl{};
    auto add = [&](const void *sp, void *dp, int esz, int ncomp) {
        for (int q = 0; q < ncomp; ++q) {
            pl.src[pl.n] = (const char *)sp + (size_t)q * c.np * esz;
            pl.dst[pl.n] = (char *)dp + (size_t)q * c.np * esz;
            pl.esz[pl.n] = esz;
            ++pl.n;
        }
    };
    if (c.prec == MHDPIC_PREC_MIXED) {
        add(src.pos, dst.pos, 16, 1);
        add(src.vel, dst.vel, 16, 1);
    } else {
        add(src.x, dst.x, 8, c.ndim);
        add(src.p64, dst.p64, 8, 3);
    }
    if (src.tinj && dst.tinj)
        add(src.tinj, dst.tinj, 8, 1);
    k_gather_all<<<grid_for(c.np, 256), 256, 0, st>>>(c.np, perm, pl);
    return 1;
}

int launch_gather_f64(int64_t np, const int32_t *perm, const double *src, double *dst, cudaStream_t st)
{
    if (np <= 0)
        return 0;
    Planes pl{};
    pl.src[0] = src;
    pl.dst[0] = dst;
    pl.esz[0] = 8;
    pl.n = 1;
    k_gather_all<<<grid_for(np, 256), 256, 0, st>>>(np, perm, pl);
    return 1;
}

namespace {
__global__ void k_clock_advance(double *clock, double dt) { clock[0] = clock[0] + dt; }
}  // namespace

int launch_clock_advance(double *clock, double dt, cudaStream_t st)
{
    k_clock_advance<<<1, 1, 0, st>>>(clock, dt);
    return 1;
}

namespace {

// Mark the slots [offset[nkeys], np) of the current set as free: after a push
// that applied a sort they still hold the states of an older step.
template <int PREC>
__global__ void k_mark_free(Ctx c, const int32_t *__restrict__ offset)
{
    const int64_t live = offset[c.nkeys];
    for (int64_t j = live + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < c.np;
         j += (int64_t)gridDim.x * blockDim.x) {
        if (PREC == MHDPIC_PREC_MIXED) {
            c.pos[j] = make_int4(DEAD_CELL, 0, 0, 0);
            c.vel[j] = make_float4(0.f, 0.f, 0.f, 0.f);
        } else {
            c.x[j] = __longlong_as_double(0x7ff8000000000000ll);
            for (int d = 0; d < 3; ++d)
                c.p64[(int64_t)d * c.np + j] = 0.0;
        }
    }
}

__global__ void k_count_live(Ctx c, int prec, unsigned long long *out)
{
    unsigned long long n = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < c.np;
         i += (int64_t)gridDim.x * blockDim.x)
        n += prec == MHDPIC_PREC_MIXED ? (c.pos[i].x != DEAD_CELL) : !isnan(c.x[i]);
    for (int o = 16; o > 0; o >>= 1)
        n += __shfl_xor_sync(0xffffffffu, n, o);
    if ((threadIdx.x & 31) == 0 && n)
        atomicAdd(out, n);
}

}  // namespace

int launch_mark_free(const Ctx &c, const SortScratch &s, cudaStream_t st)
{
    if (c.np <= 0)
        return 0;
    if (c.prec == MHDPIC_PREC_MIXED)
        k_mark_free<MHDPIC_PREC_MIXED><<<grid_for(c.np, 256), 256, 0, st>>>(c, s.offset);
    else
        k_mark_free<MHDPIC_PREC_FP64><<<grid_for(c.np, 256), 256, 0, st>>>(c, s.offset);
    return 1;
}

int launch_count_live(const Ctx &c, unsigned long long *out, cudaStream_t st)
{
    cudaMemsetAsync(out, 0, sizeof(unsigned long long), st);
    if (c.np <= 0)
        return 0;
    k_count_live<<<grid_for(c.np, 256), 256, 0, st>>>(c, c.prec, out);
    return 1;
}

int launch_max_count(const Ctx &c, const SortScratch &s, cudaStream_t st)
{
    cudaMemsetAsync(s.max_count, 0, sizeof(int32_t), st);
    k_max_count<<<grid_for(c.nkeys, 256), 256, 0, st>>>(c.nkeys, s.count, s.max_count);
    return 1;
}

}  // namespace mhdpic
