// Velocity-Verlet NVE pieces and the permutation kernels between the caller's atom
// order and the internal cell-sorted order.  Positions and velocities are fp64: at 8 M atoms
// the box is ~450 Angstrom and a 1 fs displacement (~1e-3 Angstrom) would lose most of its
// digits in fp32.
#include "common.cuh"

namespace mlip {

// Force on atom i: the fp64 array when the context evaluates in fp64, else the fp32 one.
__device__ __forceinline__ double3 load_force(const float4 *force, const double *force_d, int64_t i) {
    if (force_d) return make_double3(force_d[3 * i], force_d[3 * i + 1], force_d[3 * i + 2]);
    const float4 f = force[i];
    return make_double3(f.x, f.y, f.z);
}

// The forces that the evaluation after a move accumulates into: the kernels that move atoms clear them on the way (a separate clear is a
// launch and a pass of its own).
__device__ __forceinline__ void clear_for_eval(const EvalClear &c, int64_t i) {
    if (c.force) c.force[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (c.force_d) { c.force_d[3 * i] = 0.0; c.force_d[3 * i + 1] = 0.0; c.force_d[3 * i + 2] = 0.0; }
}

// What the drift tracks besides moving the atoms.
struct DriftArgs {
    double dt;
    CellGrid g;
    float skin_half2, trigger2, far2;
    float *disp;
    int *status, *rebuild_flag, *far_flag;
    EvalClear clear;
};
// x += dt v;  wrap into [0, L);  track the displacement since the last list build.
__device__ __forceinline__ void drift_atom(const DriftArgs &d, int64_t i, double4 p, const double (&v)[3], double4 *pos4) {
    const double px[3] = {p.x, p.y, p.z};
    double x[3];
    float d2 = 0.f;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        x[a] = fma(d.dt, v[a], px[a]);
        const float s = d.disp[3 * i + a] + (float)(d.dt * v[a]);
        d.disp[3 * i + a] = s;
        d2 += s * s;
        const double L = d.g.box[a];
        if (x[a] >= L) x[a] -= L;
        else if (x[a] < 0.0) x[a] += L;
        if (!(x[a] >= 0.0 && x[a] < L)) x[a] = 0.0;   // -eps + L rounds to L; NaN is reported below
    }
    if (!(d2 <= d.skin_half2)) atomicOr(d.status, d2 == d2 ? FLAG_SKIN_EXCEEDED : FLAG_NONFINITE);
    if (d2 > d.trigger2) *d.rebuild_flag = 1;   // same value from every writer
    if (!(d2 <= d.far2)) *d.far_flag = 1;       // from now on the lists' far entries may come inside r_cut
    pos4[i] = make_double4(x[0], x[1], x[2], p.w);
    clear_for_eval(d.clear, i);
}

// v += dt/2 a  (CLOSE: twice, the second half kick of one step and the first of the next, which see the same forces), then the drift.
// Every operation is rounded in a fixed way, so a trajectory does not depend on how it is cut into calls.
template <bool CLOSE>
__global__ void k_kick_drift(int64_t n, const double *__restrict__ mass, double4 *pos4, double *vel, const float4 *force, const double *force_d,
                             const double *vscale, DriftArgs d, unsigned long long *stamp) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    allow_next();
    wait_previous();
    stamp_begin(stamp);
    if (i >= n) return;
    const double4 p = pos4[i];
    const double3 f3 = load_force(force, force_d, i);
    const double f[3] = {f3.x, f3.y, f3.z};
    const double k = 0.5 * d.dt * ACC_UNIT / mass[(int)p.w];
    const double sc = vscale ? *vscale : 1.0;   // thermostat factor applied ahead of the kick (NVT)
    double v[3];
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        v[a] = vel[3 * i + a];
        if (CLOSE) v[a] = fma(k, f[a], v[a]);
        v[a] = fma(k, f[a], v[a] * sc);
        vel[3 * i + a] = v[a];
    }
    drift_atom(d, i, p, v, pos4);
    stamp_end(stamp);
}

// v += dt/2 a
__global__ void k_kick(int64_t n, double dt, const double *__restrict__ mass, const double4 *pos4, double *vel, const float4 *force,
                       const double *force_d, unsigned long long *stamp) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    allow_next();
    wait_previous();
    stamp_begin(stamp);
    if (i >= n) return;
    const double3 f = load_force(force, force_d, i);
    const double k = 0.5 * dt * ACC_UNIT / mass[(int)pos4[i].w];
    vel[3 * i] = fma(k, f.x, vel[3 * i]); vel[3 * i + 1] = fma(k, f.y, vel[3 * i + 1]); vel[3 * i + 2] = fma(k, f.z, vel[3 * i + 2]);
    stamp_end(stamp);
}

// Half-step (dt/2) of a Nose-Hoover chain of three thermostats coupled to the kinetic energy in acc[ACC_KINETIC]
// (Martyna-Tuckerman-Tobias-Klein factorisation, one Suzuki-Yoshida term).  One thread calls it.  state = {v_eta[3], eta[3], scale}:
//   dv_eta_k/dt = G_k - v_eta_{k+1} v_eta_k,  G_1 = (2 KE - N_f kT) / Q_1,  G_k = (Q_{k-1} v_eta_{k-1}^2 - kT) / Q_k,
//   particle velocities scale by exp(-v_eta_1 dt/2); the stored kinetic energy is scaled with them.
// (Every step of a run waits for this chain of dependent operations, twice: divisions by the thermostat masses are products with their
// reciprocals, and the exponentials, whose arguments are of the order of the step over the damping time, Taylor polynomials: below
// 1/32 the first omitted term is 2^-45 / 9! relative, 8e-20.)
struct NhcHalf { double n_f, kT, q1, qk, inv_q1, inv_qk, dt; double *state; };   // state = nullptr: no thermostat
__device__ __forceinline__ double exp_near_zero(double x) {
    if (fabs(x) > 0.03125) return exp(x);
    double y = 1.0 / 40320.0;
    y = fma(y, x, 1.0 / 5040.0); y = fma(y, x, 1.0 / 720.0); y = fma(y, x, 1.0 / 120.0); y = fma(y, x, 1.0 / 24.0);
    y = fma(y, x, 1.0 / 6.0); y = fma(y, x, 0.5); y = fma(y, x, 1.0);
    return fma(y, x, 1.0);
}
__device__ void nhc_half(const NhcHalf &h, double *acc) {
    constexpr int M = 3;
    double *state = h.state;
    double v[M] = {state[0], state[1], state[2]};
    const double q[M] = {h.q1, h.qk, h.qk}, iq[M] = {h.inv_q1, h.inv_qk, h.inv_qk}, d = 0.5 * h.dt;
    double ke2 = 2.0 * acc[ACC_KINETIC];
    double G[M];
    G[0] = (ke2 - h.n_f * h.kT) * iq[0];
    for (int c = 1; c < M; ++c) G[c] = (q[c - 1] * v[c - 1] * v[c - 1] - h.kT) * iq[c];
    v[M - 1] += 0.5 * d * G[M - 1];
    for (int c = M - 2; c >= 0; --c) {
        const double a = exp_near_zero(-0.25 * d * v[c + 1]);
        v[c] = (v[c] * a + 0.5 * d * G[c]) * a;
    }
    const double scale = exp_near_zero(-d * v[0]);
    ke2 *= scale * scale;
    for (int c = 0; c < M; ++c) state[3 + c] += d * v[c];
    G[0] = (ke2 - h.n_f * h.kT) * iq[0];
    for (int c = 0; c < M - 1; ++c) {
        const double a = exp_near_zero(-0.25 * d * v[c + 1]);
        v[c] = (v[c] * a + 0.5 * d * G[c]) * a;
        G[c + 1] = (q[c] * v[c] * v[c] - h.kT) * iq[c + 1];
    }
    v[M - 1] += 0.5 * d * G[M - 1];
    for (int c = 0; c < M; ++c) state[c] = v[c];
    state[6] = scale;
    acc[ACC_KINETIC] = 0.5 * ke2;
}

__global__ void k_scale_velocities(int64_t n3, double *vel, const double *scale, unsigned long long *stamp) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    allow_next();
    wait_previous();
    stamp_begin(stamp);
    if (i < n3) vel[i] *= *scale;
    stamp_end(stamp);
}

// Kinetic energy with a fixed summation order (grid-stride partial sums per block, then one warp of the block that finishes last
// adds the block sums in index order), so that the thermostat -- and with it an NVT trajectory -- is bit-reproducible.  What changes the
// velocities just before rides along: CHANGE = 1 the half kick that closes a step, 2 the thermostat's factor; and the thermostat half
// step that needs the energy follows in the last block.  (As kernels of their own these were eight of a step's ten launches:
// 4,394 atoms 152 us per step, of which the evaluation was 65.)
constexpr int KIN_BLOCKS = 1184;
template <int CHANGE>
__global__ void __launch_bounds__(256) k_kinetic(int64_t n, double dt, const double *__restrict__ mass, const double4 *pos4, double *vel, const float4 *force,
                                                 const double *force_d, const double *scale, double *block_sum, unsigned int *ticket, double *acc,
                                                 NhcHalf nhc, unsigned long long *stamp) {
    __shared__ double part[8];
    __shared__ bool last;
    allow_next();
    wait_previous();
    stamp_begin(stamp);
    double e = 0.0;
    const double sc = CHANGE == 2 ? *scale : 1.0;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
        double v[3] = {vel[3 * i], vel[3 * i + 1], vel[3 * i + 2]};
        const double m = mass[(int)pos4[i].w];
        if (CHANGE == 1) {
            const double3 f = load_force(force, force_d, i);
            const double k = 0.5 * dt * ACC_UNIT / m;
            v[0] = fma(k, f.x, v[0]); v[1] = fma(k, f.y, v[1]); v[2] = fma(k, f.z, v[2]);
        }
        if (CHANGE == 2) { v[0] *= sc; v[1] *= sc; v[2] *= sc; }
        if (CHANGE != 0) { vel[3 * i] = v[0]; vel[3 * i + 1] = v[1]; vel[3 * i + 2] = v[2]; }
        e = fma(0.5 * m, fma(v[2], v[2], fma(v[1], v[1], __dmul_rn(v[0], v[0]))), e);
    }
    for (int o = 16; o; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
    if ((threadIdx.x & 31) == 0) part[threadIdx.x >> 5] = e;
    __syncthreads();
    if (threadIdx.x >= 32) return;
    e = threadIdx.x < 8 ? part[threadIdx.x] : 0.0;
    for (int o = 16; o; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
    if (threadIdx.x == 0) {
        block_sum[blockIdx.x] = e;
        __threadfence();
        last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    }
    __syncwarp();
    if (!last) return;
    __threadfence();
    e = 0.0;
    for (unsigned b = threadIdx.x; b < gridDim.x; b += 32) e += *(volatile double *)(block_sum + b);
    for (int o = 16; o; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
    if (threadIdx.x == 0) {
        *ticket = 0;
        acc[ACC_KINETIC] = e * (1.0 / ACC_UNIT);
        if (nhc.state) nhc_half(nhc, acc);
        stamp_end(stamp);
    }
}

// What lies between two evaluations of an NVT run in one launch, for systems that a cluster holds with an atom per thread: the half kick that
// closes a step, the two thermostat half steps (each after the kinetic energy of the velocities as they stand), the next step's
// half kick and drift.  The sums are taken in k_kinetic's order -- groups of 256 atoms, then the groups' sums -- and the blocks meet at the
// hardware barrier of the cluster.  4,394 atoms: three launches were 12 us of a step's 61 and the gaps between
// them 9; this one takes 9.
constexpr int NVT_CTA = 1024, NVT_CLUSTER = 8;
__device__ __forceinline__ void cluster_sync_all() {
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__global__ void __launch_bounds__(NVT_CTA) k_nvt_between(int n, const double *__restrict__ mass, double4 *pos4, double *vel, const float4 *force,
                                                        const double *force_d, double *block_sum, double *acc, NhcHalf nhc, DriftArgs d,
                                                        unsigned long long *stamp) {
    __shared__ double part[NVT_CTA / 32];
    const int i = blockIdx.x * NVT_CTA + threadIdx.x, lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    allow_next();
    wait_previous();
    stamp_begin(stamp);
    double4 p = make_double4(0.0, 0.0, 0.0, 0.0);
    double v[3] = {0.0, 0.0, 0.0}, f[3] = {0.0, 0.0, 0.0}, m = 0.0, k = 0.0;
    if (i < n) {
        p = pos4[i];
        const double3 f3 = load_force(force, force_d, i);
        f[0] = f3.x; f[1] = f3.y; f[2] = f3.z;
        m = mass[(int)p.w];
        k = 0.5 * d.dt * ACC_UNIT / m;
#pragma unroll
        for (int a = 0; a < 3; ++a) v[a] = fma(k, f[a], vel[3 * i + a]);
    }
    double sc = 1.0;
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
#pragma unroll
        for (int a = 0; a < 3; ++a) v[a] *= sc;
        double e = fma(0.5 * m, fma(v[2], v[2], fma(v[1], v[1], __dmul_rn(v[0], v[0]))), 0.0);
        for (int o = 16; o; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
        if (lane == 0) part[warp] = e;
        __syncthreads();
        if (threadIdx.x < NVT_CTA / 256) {
            const double *q = part + 8 * threadIdx.x;
            const int b = blockIdx.x * (NVT_CTA / 256) + threadIdx.x;
            if (256 * b < n) block_sum[b] = ((q[0] + q[4]) + (q[2] + q[6])) + ((q[1] + q[5]) + (q[3] + q[7]));
        }
        cluster_sync_all();
        if (blockIdx.x == 0 && warp == 0) {
            double s = 0.0;
            for (int b = lane; 256 * b < n; b += 32) s += *(volatile double *)(block_sum + b);
            for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
            if (lane == 0) {
                acc[ACC_KINETIC] = s * (1.0 / ACC_UNIT);
                nhc_half(nhc, acc);
            }
        }
        cluster_sync_all();
        sc = *(volatile double *)(nhc.state + 6);
    }
    if (i < n) {
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            v[a] = fma(k, f[a], v[a] * sc);
            vel[3 * i + a] = v[a];
        }
        drift_atom(d, i, p, v, pos4);
    }
    stamp_end(stamp);
}

// Per-atom outputs in the caller's order, and the totals: one launch.  FIN: float4, or double for three per atom.
template <typename FIN, typename EIN, typename FOUT>
__global__ void k_outputs(int64_t n, const int32_t *__restrict__ user_of, const FIN *force, const EIN *e_in,
                          FOUT *__restrict__ forces_out, FOUT *__restrict__ e_atom, const double *acc, double *__restrict__ energy,
                          double *__restrict__ virial) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    wait_previous();
    if (i == 0) {
        if (energy) *energy = acc[ACC_ENERGY];
        if (virial)
            for (int q = 0; q < 9; ++q) virial[q] = acc[ACC_VIRIAL + q];
    }
    if (i >= n || !(forces_out || e_atom)) return;
    const int64_t u = user_of[i];
    if (forces_out) {
        if constexpr (sizeof(FIN) == sizeof(float4)) {
            const float4 f = force[i];
            forces_out[3 * u] = (FOUT)f.x; forces_out[3 * u + 1] = (FOUT)f.y; forces_out[3 * u + 2] = (FOUT)f.z;
        } else {
#pragma unroll
            for (int q = 0; q < 3; ++q) forces_out[3 * u + q] = (FOUT)force[3 * i + q];
        }
    }
    if (e_atom) e_atom[u] = (FOUT)e_in[i];
}

__global__ void k_set_positions(int64_t n, const int32_t *__restrict__ user_of, const double *pos,
                                CellGrid g, float skin_half2, double4 *pos4, float *disp, int *status,
                                float far2, int *far_flag, EvalClear clear) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    allow_next();
    wait_previous();
    if (i >= n) return;
    clear_for_eval(clear, i);
    const int64_t u = user_of[i];
    double4 p = pos4[i];
    const double x[3] = {pos[3 * u], pos[3 * u + 1], pos[3 * u + 2]};
    const double old[3] = {p.x, p.y, p.z};
    float d2 = 0.f;
    bool ok = true;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        ok = ok && (x[a] >= 0.0 && x[a] < g.box[a]);
        float d = disp[3 * i + a] + (float)min_image(x[a] - old[a], g.box[a], g.half[a]);
        disp[3 * i + a] = d;
        d2 += d * d;
    }
    if (!ok) atomicOr(status, FLAG_NONFINITE);
    else if (!(d2 <= skin_half2)) atomicOr(status, FLAG_SKIN_EXCEEDED);
    if (!(d2 <= far2)) *far_flag = 1;
    pos4[i] = make_double4(x[0], x[1], x[2], p.w);
}

__global__ void k_set_velocities(int64_t n, const int32_t *__restrict__ user_of, const double *__restrict__ vel_in,
                                 double *__restrict__ vel) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int64_t u = user_of[i];
    vel[3 * i] = vel_in[3 * u]; vel[3 * i + 1] = vel_in[3 * u + 1]; vel[3 * i + 2] = vel_in[3 * u + 2];
}

__global__ void k_get_state(int64_t n, const int32_t *__restrict__ user_of, const double4 *__restrict__ pos4,
                            const double *__restrict__ vel, double *__restrict__ pos_out, double *__restrict__ vel_out) {
    int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    const int64_t u = user_of[i];
    if (pos_out) { double4 p = pos4[i]; pos_out[3 * u] = p.x; pos_out[3 * u + 1] = p.y; pos_out[3 * u + 2] = p.z; }
    if (vel_out) { vel_out[3 * u] = vel[3 * i]; vel_out[3 * u + 1] = vel[3 * i + 1]; vel_out[3 * u + 2] = vel[3 * i + 2]; }
}

static inline unsigned nb(int64_t n) { return (unsigned)((n + 255) / 256); }
static inline float skin_half2(const mlip_ctx *c) { float h = 0.5f * (float)c->cfg.skin; return h * h; }
// Far entries lie beyond r_cut + skin / 2 at build time; a pair closes by at most twice the largest displacement, so they
// stay outside r_cut while every atom has moved less than skin / 4 (0.245: room for the fp32 bookkeeping).
static inline float far_trigger2(const mlip_ctx *c) { float h = 0.245f * (float)c->cfg.skin; return h * h; }

// The forces of the next evaluation, to be cleared by the kernel that takes this, which must be the last before it that reads them.
EvalClear eval_clear(mlip_ctx *c) {
    c->force_cleared = true;
    const bool f64 = c->cfg.precision == 1;
    return EvalClear{f64 || c->cfg.force_mode == 1 ? nullptr : c->force, f64 ? c->force_d : nullptr};
}
static NhcHalf nhc_args(mlip_ctx *c, double dt, bool thermostat) {
    return NhcHalf{c->nhc_nf, c->nhc_kT, c->nhc_q1, c->nhc_qk, 1.0 / c->nhc_q1, 1.0 / c->nhc_qk, dt, thermostat ? c->nhc : nullptr};
}
static DriftArgs drift_args(mlip_ctx *c, double dt) {
    return DriftArgs{dt, c->grid, skin_half2(c), 0.64f * skin_half2(c), far_trigger2(c), c->disp, c->status, c->rebuild_flag, c->far_flag, eval_clear(c)};
}
int launch_kick_drift(mlip_ctx *c, double dt, bool close_step, cudaStream_t s, const double *vscale) {
    unsigned long long *stamp = timed_begin(c, MARK_INTEGRATE, s);
    MLIP_CUDA_TRY(c, launch_after(close_step ? k_kick_drift<true> : k_kick_drift<false>, nb(c->n), 256, 0, s, c->n, c->mass, c->pos4, c->vel, c->force,
                                  c->force_d, vscale, drift_args(c, dt), stamp));
    timed_end(c, MARK_INTEGRATE, s);
    c->launches += 1;
    return MLIP_OK;
}
// Everything between two evaluations of an NVT run.
int launch_nvt_between(mlip_ctx *c, double dt, cudaStream_t s) {
    int rc;
    if (c->n > NVT_CTA * NVT_CLUSTER) {
        if ((rc = launch_kinetic(c, 1, true, dt, s)) != MLIP_OK || (rc = launch_kinetic(c, 2, true, dt, s)) != MLIP_OK) return rc;
        return launch_kick_drift(c, dt, false, s, c->nhc + 6);
    }
    int blocks = 1;
    while (blocks * NVT_CTA < c->n) blocks *= 2;
    const NhcHalf nhc = nhc_args(c, dt, true);
    unsigned long long *stamp = timed_begin(c, MARK_INTEGRATE, s);
    cudaLaunchAttribute attr[2] = {};
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = blocks; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(blocks); cfg.blockDim = dim3(NVT_CTA); cfg.stream = s; cfg.attrs = attr; cfg.numAttrs = 2;
    MLIP_CUDA_TRY(c, cudaLaunchKernelEx(&cfg, k_nvt_between, (int)c->n, (const double *)c->mass, c->pos4, c->vel, (const float4 *)c->force,
                                        (const double *)c->force_d, c->kin_part, c->acc, nhc, drift_args(c, dt), stamp));
    timed_end(c, MARK_INTEGRATE, s);
    c->launches += 1;
    return MLIP_OK;
}
int launch_kick(mlip_ctx *c, double dt, cudaStream_t s) {
    unsigned long long *stamp = timed_begin(c, MARK_INTEGRATE, s);
    MLIP_CUDA_TRY(c, launch_after(k_kick, nb(c->n), 256, 0, s, c->n, dt, c->mass, c->pos4, c->vel, c->force, c->force_d, stamp));
    timed_end(c, MARK_INTEGRATE, s);
    c->launches += 1;
    return MLIP_OK;
}
int launch_scale_velocities(mlip_ctx *c, cudaStream_t s) {
    unsigned long long *stamp = timed_begin(c, MARK_INTEGRATE, s);
    MLIP_CUDA_TRY(c, launch_after(k_scale_velocities, nb(3 * c->n), 256, 0, s, 3 * c->n, c->vel, c->nhc + 6, stamp));
    timed_end(c, MARK_INTEGRATE, s);
    c->launches += 1;
    return MLIP_OK;
}
int launch_kinetic(mlip_ctx *c, int change, bool thermostat, double dt, cudaStream_t s) {
    const int64_t blocks = nb(c->n) > KIN_BLOCKS ? KIN_BLOCKS : nb(c->n);
    const NhcHalf nhc = nhc_args(c, dt, thermostat);
    unsigned long long *stamp = thermostat ? timed_begin(c, MARK_INTEGRATE, s) : nullptr;
    MLIP_CUDA_TRY(c, launch_after(change == 1 ? k_kinetic<1> : change == 2 ? k_kinetic<2> : k_kinetic<0>, (unsigned)blocks, 256, 0, s, c->n, dt, c->mass,
                                  c->pos4, c->vel, c->force, c->force_d, c->nhc + 6, c->kin_part, reinterpret_cast<unsigned int *>(c->kin_part + KIN_BLOCKS),
                                  c->acc, nhc, stamp));
    if (thermostat) timed_end(c, MARK_INTEGRATE, s);
    c->launches += 1;
    return MLIP_OK;
}
int launch_outputs(mlip_ctx *c, float *forces, float *e_atom, double *energy, double *virial, cudaStream_t s) {
    const unsigned blocks = forces || e_atom ? nb(c->n) : 1;
    if (c->cfg.precision == 1)
        MLIP_CUDA_TRY(c, launch_after(k_outputs<double, double, float>, blocks, 256, 0, s, c->n, c->user_of, c->force_d, c->e_atom_d, forces, e_atom, c->acc, energy, virial));
    else
        MLIP_CUDA_TRY(c, launch_after(k_outputs<float4, float, float>, blocks, 256, 0, s, c->n, c->user_of, c->force, c->e_atom, forces, e_atom, c->acc, energy, virial));
    c->launches += 1;
    return MLIP_OK;
}
int launch_outputs_f64(mlip_ctx *c, double *forces, double *e_atom, double *energy, double *virial, cudaStream_t s) {
    const unsigned blocks = forces || e_atom ? nb(c->n) : 1;
    MLIP_CUDA_TRY(c, launch_after(k_outputs<double, double, double>, blocks, 256, 0, s, c->n, c->user_of, c->force_d, c->e_atom_d, forces, e_atom, c->acc, energy, virial));
    c->launches += 1;
    return MLIP_OK;
}
int launch_set_positions(mlip_ctx *c, const double *pos, cudaStream_t s) {
    MLIP_CUDA_TRY(c, launch_after(k_set_positions, nb(c->n), 256, 0, s, c->n, c->user_of, pos, c->grid, skin_half2(c), c->pos4, c->disp, c->status,
                                  far_trigger2(c), c->far_flag, eval_clear(c)));
    c->launches += 1;
    return MLIP_OK;
}
int launch_set_velocities(mlip_ctx *c, const double *vel, cudaStream_t s) {
    k_set_velocities<<<nb(c->n), 256, 0, s>>>(c->n, c->user_of, vel, c->vel);
    c->launches += 1;
    MLIP_CUDA_TRY(c, cudaGetLastError());
    return MLIP_OK;
}
int launch_get_state(mlip_ctx *c, double *pos, double *vel, cudaStream_t s) {
    k_get_state<<<nb(c->n), 256, 0, s>>>(c->n, c->user_of, c->pos4, c->vel, pos, vel);
    c->launches += 1;
    MLIP_CUDA_TRY(c, cudaGetLastError());
    return MLIP_OK;
}

}  // namespace mlip
