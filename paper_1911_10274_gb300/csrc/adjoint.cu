// adjoint.cu -- reverse-mode derivative of a rollout with respect to the
// actuation amplitudes and phases (gradient-based design of actuated robots).
//
// Forward: the ordinary step (Titan Sec. III-B, Eq. 1; Sec. III-A contact,
// friction and constraints) with L = L0 (1 + A sin(2 pi f t + phi)).  The
// rollout runs forward once, keeping every state if they fit (titan_adjoint_limit),
// else the state every `every` steps (checkpoints) and the states of the last
// segment; earlier segments are recomputed from their checkpoints.  Then, from
// the last step back, k_adj_step reverses one step per launch, per mass:
//   - the adjoint of x' = x + v' dt, v' = v + a dt and a = F/m + g +
//     contact/friction (the branch the forward step took at each kink), giving
//     dJ/dF and the direct terms of dJ/dx, dJ/dv;
//   - its SELL row in the forward's fixed order: each spring's adjoint seen
//     from this end (both ends compute the same spring scalars), added to this
//     mass only; the half-edge of the spring's first end also adds to the
//     spring's gradient (one owner: no atomics, a fixed summation order);
//   - dJ/dF of the step before, which its neighbours gather in the next launch.
#include <math.h>

#include <algorithm>
#include <cmath>
#include <mutex>
#include <string>
#include <vector>

#include "context_id.h"
#include "physics.cuh"
#include "sim_internal.h"

namespace {

constexpr int kT = 256;
constexpr uint32_t kOwner = 0x80000000u;
constexpr int kAdjT = 128;

// The adjoint a force on a mass carries, from (x_b, v_b) of the state after the step:
// v' = v + (F / m + ...) dt and x' = x + v' dt.  None on a fixed mass, whatever its own
// adjoint is (its neighbours must not take an infinity or NaN times 0 from it).
__device__ __forceinline__ float4 force_adjoint(float4 xo, float4 vo, float im, float dt) {
    if (im == 0.f) return make_float4(0.f, 0.f, 0.f, 0.f);
    const float vtx = vo.x + dt * xo.x, vty = vo.y + dt * xo.y, vtz = vo.z + dt * xo.z;
    return make_float4(dt * vtx * im, dt * vty * im, dt * vtz * im, 0.f);
}

// The mass part of reversing a step at state (p, v): from (xo, vo), the adjoint
// of the state after it, the direct terms (x_b, v_b) and the force's adjoint F.
template <bool GROUND>
__device__ __forceinline__ void adj_mass(const float4 &p, const float4 &v, const float4 &xo, const float4 &vo,
                                         const titan::StepConst &c, float4 &x_b, float4 &v_b, float4 &F) {
    const float im = p.w;
    x_b = make_float4(xo.x, xo.y, xo.z, 0.f);
    if (im == 0.f) {                       // fixed: x' = x, v' = 0
        v_b = F = make_float4(0.f, 0.f, 0.f, 0.f);
        return;
    }
    const float dt = c.dt;
    const float vtx = vo.x + dt * xo.x, vty = vo.y + dt * xo.y, vtz = vo.z + dt * xo.z;
    v_b = make_float4(vtx, vty, vtz, 0.f);
    F = force_adjoint(xo, vo, im, dt);
    if (GROUND && p.z < 0.f) {
        const float abx = dt * vtx, aby = dt * vty, abz = dt * vtz;
        x_b.z += -c.ground_k * im * abz;                   // a_z += kg (-z) / m
        const float vt = sqrtf(v.x * v.x + v.y * v.y);
        if (vt > 0.f) {
            const float an = c.ground_k * (-p.z) * im;
            const bool capped = vt / c.dt < c.mu * an;      // the forward's fminf choice
            const float fr = capped ? vt / c.dt : c.mu * an;
            const float wx = v.x / vt, wy = v.y / vt;
            const float frb = -(abx * wx + aby * wy);      // a_t -= fr w
            const float wbx = -fr * abx, wby = -fr * aby;
            float vtb = 0.f;
            if (!capped) x_b.z += -c.mu * c.ground_k * im * frb;
            else vtb = frb / c.dt;
            const float wdot = wbx * wx + wby * wy;
            v_b.x += (wbx - wdot * wx) / vt + vtb * wx;
            v_b.y += (wby - wdot * wy) / vt + vtb * wy;
        }
    }
}

// The adjoint of one spring seen from the mass at (p, v): adds to x_b, v_b and
// returns dJ/dL.  a = {k, L0, A cos phi, A sin phi}, sc the step's (sin, cos)
// of the clock phase.  A padding entry is a spring of the mass to itself.
__device__ __forceinline__ float adj_half_edge(const float4 &p, const float4 &v, const float4 &Fi, const float4 &q,
                                               const float4 &w, const float4 &Fj, const float4 &a, float2 sc, float cd,
                                               float4 &x_b, float4 &v_b) {
    const float dx = q.x - p.x, dy = q.y - p.y, dz = q.z - p.z;
    const float l2 = dx * dx + dy * dy + dz * dz;
    if (!(l2 > 0.f)) return 0.f;                          // zero length: no force
    const float inv = rsqrtf(l2);
    const float l = l2 * inv;
    const float ux = dx * inv, uy = dy * inv, uz = dz * inv;
    const float k = a.x;
    const float L = a.y + a.y * (a.z * sc.x + a.w * sc.y);
    const float dvx = w.x - v.x, dvy = w.y - v.y, dvz = w.z - v.z;
    const float rate = dvx * ux + dvy * uy + dvz * uz;
    const float f = k * (l - L) + cd * rate;
    const float gx = Fi.x - Fj.x, gy = Fi.y - Fj.y, gz = Fi.z - Fj.z;
    const float fb = gx * ux + gy * uy + gz * uz;
    const float lb = k * fb, rb = cd * fb;
    const float ubx = f * gx + rb * dvx, uby = f * gy + rb * dvy, ubz = f * gz + rb * dvz;
    v_b.x -= rb * ux; v_b.y -= rb * uy; v_b.z -= rb * uz;
    const float udot = ubx * ux + uby * uy + ubz * uz;
    x_b.x -= (ubx - udot * ux) * inv + lb * ux;
    x_b.y -= (uby - udot * uy) * inv + lb * uy;
    x_b.z -= (ubz - udot * uz) * inv + lb * uz;
    return -lb;
}

// One reversed step: the mass part of this thread's mass, then its row, then
// the force adjoint of the step before (Fout; the neighbours' is read from Fin).
// (xb, vb) are this mass's alone and updated in place.
//
// Bound by the latency of the row stream (20 bytes an entry from L2) and of the
// gathers (48 bytes an entry; L1 serves 60 % of all sectors, the masses of 2,500
// threads and their neighbours just filling it).  Two entries are reversed per iteration, with the next
// two's constants already requested; 128-thread blocks, six per SM.  The row
// stream through an asynchronous ring in shared memory measured 9 % slower (it
// takes L1 from the gathers), adding to the sums by load and store 6 %.  The sine
// and cosine of each spring's own phase are in the row and the clock's come with
// the launch, so no trigonometric function is left in the loop: the spring's
// (dJ/dA, dJ/dphi) is a rotation of the two sums kept here, formed once at the
// end (k_adj_gather).  256 robots, 107,193 masses: a mass and a spring kernel per
// step 44 us, this 18.
template <bool HAS_C, bool GROUND>
__global__ void __launch_bounds__(kAdjT, 6)
k_adj_step(const MassState *__restrict__ X, const float4 *__restrict__ Fin, float4 *__restrict__ Fout,
           float4 *__restrict__ xb, float4 *__restrict__ vb, uint32_t n, const uint32_t *__restrict__ slice_off,
           const uint32_t *__restrict__ nbr, const float4 *__restrict__ row, const float *__restrict__ cc,
           titan::StepConst c, float2 sc, float2 *__restrict__ gacc) {
    const uint32_t tid = threadIdx.x, i = blockIdx.x * kAdjT + tid;
    if (i >= n) return;
    const uint32_t sl = i >> 5;
    uint32_t e = slice_off[sl] + (i & 31);
    const uint32_t end = slice_off[sl + 1];               // widths are even
    float4 p, v, x_b, v_b, Fi;
    titan::load_state(X + i, p, v);
    adj_mass<GROUND>(p, v, xb[i], vb[i], c, x_b, v_b, Fi);
    uint32_t nj0, nj1;
    float4 na0, na1;
    auto request = [&](uint32_t x) {
        if (x < end) {
            nj0 = __ldcg(nbr + x);
            nj1 = __ldcg(nbr + x + 32);
            na0 = __ldcg(row + x);
            na1 = __ldcg(row + x + 32);
        }
    };
    request(e);
    for (; e < end; e += 64) {
        const uint32_t j0 = nj0, j1 = nj1;
        const float4 a0 = na0, a1 = na1;
        request(e + 64);
        const uint32_t i0 = j0 & ~kOwner, i1 = j1 & ~kOwner;
        const bool own0 = j0 & kOwner, own1 = j1 & kOwner;
        float4 q0, w0, q1, w1;
        titan::load_state(X + i0, q0, w0);
        titan::load_state(X + i1, q1, w1);
        const float4 F0 = __ldg(Fin + i0), F1 = __ldg(Fin + i1);
        const float c0 = HAS_C ? __ldcg(cc + e) : c.c_uniform, c1 = HAS_C ? __ldcg(cc + e + 32) : c.c_uniform;
        const float L0 = adj_half_edge(p, v, Fi, q0, w0, F0, a0, sc, c0, x_b, v_b);
        const float L1 = adj_half_edge(p, v, Fi, q1, w1, F1, a1, sc, c1, x_b, v_b);
        // one owner per entry and launch: no order is left open, and nothing is waited for
        if (own0) atomicAdd(gacc + e, make_float2(L0 * sc.x, L0 * sc.y));
        if (own1) atomicAdd(gacc + e + 32, make_float2(L1 * sc.x, L1 * sc.y));
    }
    xb[i] = x_b;
    vb[i] = v_b;
    Fout[i] = force_adjoint(x_b, v_b, p.w, c.dt);
}

// The rows of the reverse pass: {k, L0, A cos phi, A sin phi} per entry.
__global__ void k_adj_rows(const float2 *__restrict__ kl, const float2 *__restrict__ act, uint32_t n,
                           float4 *__restrict__ row) {
    const uint32_t e = blockIdx.x * kT + threadIdx.x;
    if (e >= n) return;
    const float2 a = kl[e], s = act[e];
    float sn, cs;
    sincosf(s.y, &sn, &cs);
    row[e] = make_float4(a.x, a.y, s.x * cs, s.x * sn);
}

// Spring q's gradient from the sums (P, Q) of dJ/dL sin(clock), dJ/dL cos(clock)
// kept at its owner entry: L = L0 (1 + A sin(clock + phi)).
__global__ void k_adj_gather(const float2 *__restrict__ gacc, const uint32_t *__restrict__ owner,
                             const float2 *__restrict__ kl, const float2 *__restrict__ act, uint32_t S,
                             float *__restrict__ grad_amp, float *__restrict__ grad_phase) {
    const uint32_t q = blockIdx.x * kT + threadIdx.x;
    if (q >= S) return;
    const uint32_t e = owner[q];
    const float2 g = gacc[e], s = act[e];
    const float L0 = kl[e].y;
    float sn, cs;
    sincosf(s.y, &sn, &cs);
    grad_amp[q] = L0 * (g.x * cs + g.y * sn);
    grad_phase[q] = L0 * s.x * (g.y * cs - g.x * sn);
}

__global__ void k_adj_seed(const float *__restrict__ seed_pos, const float *__restrict__ seed_vel,
                           const uint32_t *__restrict__ dev_of_caller, uint32_t n, float4 *__restrict__ xb,
                           float4 *__restrict__ vb) {
    const uint32_t i = blockIdx.x * kT + threadIdx.x;
    if (i >= n) return;
    const uint32_t d = dev_of_caller[i];
    xb[d] = make_float4(seed_pos[3 * (size_t)i], seed_pos[3 * (size_t)i + 1], seed_pos[3 * (size_t)i + 2], 0.f);
    if (seed_vel)
        vb[d] = make_float4(seed_vel[3 * (size_t)i], seed_vel[3 * (size_t)i + 1], seed_vel[3 * (size_t)i + 2], 0.f);
}

__global__ void k_adj_force0(const MassState *__restrict__ X, const float4 *__restrict__ xb,
                             const float4 *__restrict__ vb, uint32_t n, float dt, float4 *__restrict__ F) {
    const uint32_t i = blockIdx.x * kT + threadIdx.x;
    if (i < n) F[i] = force_adjoint(xb[i], vb[i], X[i].p.w, dt);
}

// The workspaces of titan_adjoint come from a pool of the library's own per
// device, stream-ordered like the default pool but keeping up to kAdjKeep
// between calls (the default pool gives every byte back at each
// synchronisation, and mapping them again took as long as dozens of steps).
// adjoint_trim gives the memory back (titan_destroy); before that the driver takes
// it for any allocation that needs it.
constexpr uint64_t kAdjKeep = 2ull << 30;
// Kept while the device's context lives (a cudaDeviceReset destroys it); the device's
// default pool serves where that cannot be told.
struct Pool {
    unsigned long long ctx_id = 0;
    cudaMemPool_t pool = nullptr;
};
std::mutex g_pool_mu;
Pool g_pool[64];

cudaError_t adjoint_pool(int dev, cudaMemPool_t *out) {
    if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(g_pool_mu);
    const unsigned long long id = titan::current_context_id();
    if (id == 0) return cudaDeviceGetDefaultMemPool(out, dev);
    if (!g_pool[dev].pool || !titan::same_context(g_pool[dev].ctx_id, id)) {
        cudaMemPoolProps props = {};
        props.allocType = cudaMemAllocationTypePinned;
        props.location.type = cudaMemLocationTypeDevice;
        props.location.id = dev;
        cudaMemPool_t p = nullptr;
        cudaError_t e = cudaMemPoolCreate(&p, &props);
        if (e != cudaSuccess) return e;
        uint64_t keep = kAdjKeep;
        e = cudaMemPoolSetAttribute(p, cudaMemPoolAttrReleaseThreshold, &keep);
        if (e != cudaSuccess) {
            cudaMemPoolDestroy(p);
            return e;
        }
        g_pool[dev] = {id, p};
    }
    *out = g_pool[dev].pool;
    return cudaSuccess;
}

titan_status afail(titan_sim *sim, titan_status st, const std::string &msg) {
    sim->error = msg;
    return st;
}

#define ADJ_CK(call)                                                                               \
    do {                                                                                           \
        cudaError_t e_ = (call);                                                                   \
        if (e_ != cudaSuccess) {                                                                   \
            st_ = afail(sim, e_ == cudaErrorMemoryAllocation ? TITAN_E_OOM : TITAN_E_CUDA,         \
                        std::string(#call) + ": " + cudaGetErrorString(e_));                        \
            cudaGetLastError();                                                                    \
            goto done;                                                                             \
        }                                                                                          \
    } while (0)

}  // namespace

void titan::adjoint_trim(int dev) {
    std::lock_guard<std::mutex> lk(g_pool_mu);
    if (dev >= 0 && dev < 64 && g_pool[dev].pool && same_context(g_pool[dev].ctx_id, current_context_id()))
        cudaMemPoolTrimTo(g_pool[dev].pool, 0);
}

extern "C" titan_status titan_adjoint_limit(titan_sim *sim, uint64_t bytes) {
    if (!sim) return TITAN_E_INVALID;
    if (sim->busy.exchange(true)) return afail(sim, TITAN_E_BUSY, "another call on this handle is in progress");
    sim->adj_limit = bytes;
    sim->busy.store(false);
    return TITAN_OK;
}

extern "C" titan_status titan_adjoint(titan_sim *sim, uint64_t n_steps, uint32_t every,
                                      const float *seed_pos_dev, const float *seed_vel_dev,
                                      float *grad_amp_dev, float *grad_phase_dev) {
    if (!sim) return TITAN_E_INVALID;
    if (sim->busy.exchange(true)) return afail(sim, TITAN_E_BUSY, "another call on this handle is in progress");
    titan_status st_ = TITAN_OK;
    int prev = -1;
    const uint32_t nd = sim->n_dev, S = sim->s;
    const size_t state_bytes = (size_t)std::max(nd, 1u) * sizeof(MassState);
    const size_t vec_bytes = (size_t)std::max(nd, 1u) * sizeof(float4);
    cudaStream_t s = sim->stream;
    MassState *ckpt = nullptr, *seg = nullptr;
    float4 *xb = nullptr, *vb = nullptr, *Fb[2] = {nullptr, nullptr}, *row = nullptr;
    long long *seg_steps = nullptr;
    float2 *gacc = nullptr;
    cudaMemPool_t pool = nullptr;
    uint64_t n_seg = 0;
    int cur = 0;
    if ((st_ = titan::ensure_layout(sim)) != TITAN_OK) goto out;
    if (sim->accumulate != TITAN_ACCUM_CSR) { st_ = afail(sim, TITAN_E_UNSUPPORTED, "the adjoint needs the CSR (deterministic) accumulation"); goto out; }
    if (sim->act_mode == 2) { st_ = afail(sim, TITAN_E_UNSUPPORTED, "the adjoint differentiates the sinusoidal actuation (mode 1) only"); goto out; }
    if (!sim->has_act) { st_ = afail(sim, TITAN_E_INVALID, "the adjoint differentiates the actuation: call titan_set_actuation first"); goto out; }
    if (!seed_pos_dev || (S && (!grad_amp_dev || !grad_phase_dev))) { st_ = afail(sim, TITAN_E_INVALID, "null seed or gradient array"); goto out; }
    if (every == 0) every = 50;
    cudaGetDevice(&prev);
    if (cudaSetDevice(sim->device) != cudaSuccess) { st_ = afail(sim, TITAN_E_CUDA, "cannot select the device"); goto out; }
    {
        const uint32_t E = sim->sell.entries;
        // per entry the neighbour and whether this end owns the spring's gradient (built once)
        if (!sim->d_adj_nbr) {
            std::vector<uint32_t> nb(sim->sell.nbr);
            nb.resize(std::max<size_t>(E, 1), 0);
            std::vector<uint32_t> owner(S);
            for (uint32_t q = 0; q < S; ++q) {
                owner[q] = sim->sell.entry_of_end[2 * (size_t)q];
                nb[owner[q]] |= kOwner;
            }
            void *p1 = nullptr, *p2 = nullptr;
            ADJ_CK(cudaMalloc(&p1, nb.size() * 4));
            sim->allocations.push_back(p1);
            ADJ_CK(cudaMalloc(&p2, std::max<size_t>(owner.size(), 1) * 4));
            sim->allocations.push_back(p2);
            ADJ_CK(cudaMemcpy(p1, nb.data(), nb.size() * 4, cudaMemcpyHostToDevice));
            ADJ_CK(cudaMemcpy(p2, owner.data(), owner.size() * 4, cudaMemcpyHostToDevice));
            sim->d_adj_nbr = static_cast<uint32_t *>(p1);
            sim->d_adj_owner = static_cast<uint32_t *>(p2);
        }
        const unsigned gm = (nd + kT - 1) / kT, ga = (nd + kAdjT - 1) / kAdjT;
        ADJ_CK(adjoint_pool(sim->device, &pool));
        auto take = [&](auto **p, size_t bytes) { return cudaMallocFromPoolAsync((void **)p, bytes, pool, s); };
        ADJ_CK(take(&xb, vec_bytes));
        ADJ_CK(take(&vb, vec_bytes));
        for (int b = 0; b < 2; ++b) ADJ_CK(take(&Fb[b], vec_bytes));
        ADJ_CK(take(&gacc, std::max<size_t>(E, 1) * sizeof(float2)));
        ADJ_CK(take(&row, std::max<size_t>(E, 1) * sizeof(float4)));
        // the states: all of them in one segment, or, if that is too much or the device has no
        // room for it, segments of `every` steps
        uint64_t len_max = 0;
        auto keep = [&](bool whole) {
            len_max = whole ? n_steps : std::min<uint64_t>(every, n_steps);
            n_seg = n_steps ? (n_steps + len_max - 1) / len_max : 0;
            cudaError_t e = n_seg > 1 ? take(&ckpt, state_bytes * (n_seg - 1)) : cudaSuccess;
            if (e == cudaSuccess) e = take(&seg, state_bytes * (len_max + 1));
            if (e == cudaSuccess) e = take(&seg_steps, sizeof(long long) * (len_max + 1));
            return e;
        };
        bool whole = n_steps < sim->adj_limit / state_bytes;       // n_steps + 1 states
        if (whole) {
            const cudaError_t room = keep(true);
            whole = !(room == cudaErrorMemoryAllocation && n_steps > every);
            if (whole) ADJ_CK(room);
        }
        if (!whole) {
            cudaGetLastError();
            if (seg) cudaFreeAsync(seg, s);           // taken for the whole trajectory before the room ran out
            seg = nullptr;
            ADJ_CK(keep(false));
        }
        ADJ_CK(cudaMemsetAsync(gacc, 0, std::max<size_t>(E, 1) * sizeof(float2), s));
        if (E) {
            k_adj_rows<<<(E + kT - 1) / kT, kT, 0, s>>>(sim->d_kl, sim->d_act, E, row);
            ADJ_CK(cudaGetLastError());
        }
        const uint64_t step0 = sim->steps;
        // forward rollout through the ordinary step, keeping a checkpoint at the start of every
        // segment but the last, whose states are all kept as they are formed
        for (uint64_t g = 0; g < n_seg; ++g) {
            const uint64_t len = std::min<uint64_t>(len_max, n_steps - g * len_max);
            const bool last = g + 1 == n_seg;
            ADJ_CK(cudaMemcpyAsync(last ? seg : ckpt + g * nd, sim->state[sim->cur], state_bytes, cudaMemcpyDeviceToDevice, s));
            if (!last) {
                for (uint64_t k = 0; k < len; ++k) {
                    ADJ_CK(titan::enqueue_sim_step(sim, s, sim->cur, k > 0));
                    sim->cur ^= 1;
                    ++sim->steps;
                }
                continue;
            }
            ADJ_CK(cudaMemcpyAsync(seg_steps, sim->steps_dev + sim->cur, sizeof(long long), cudaMemcpyDeviceToDevice, s));
            for (uint64_t k = 0; k < len; ++k)
                ADJ_CK(titan::enqueue_sim_step_io(sim, s, seg + k * nd, seg + (k + 1) * nd, seg_steps + k,
                                                  seg_steps + k + 1, k > 0));
            ADJ_CK(cudaMemcpyAsync(sim->state[sim->cur], seg + len * nd, state_bytes, cudaMemcpyDeviceToDevice, s));
            ADJ_CK(cudaMemcpyAsync(sim->steps_dev + sim->cur, seg_steps + len, sizeof(long long), cudaMemcpyDeviceToDevice, s));
            sim->steps += len;
        }
        // seed dJ/dx_T, dJ/dv_T in device order; gradients start at zero
        ADJ_CK(cudaMemsetAsync(xb, 0, vec_bytes, s));
        ADJ_CK(cudaMemsetAsync(vb, 0, vec_bytes, s));
        if (sim->n) {
            k_adj_seed<<<(sim->n + kT - 1) / kT, kT, 0, s>>>(seed_pos_dev, seed_vel_dev, sim->d_dev_of_caller,
                                                             sim->n, xb, vb);
            ADJ_CK(cudaGetLastError());
            k_adj_force0<<<gm, kT, 0, s>>>(sim->state[sim->cur], xb, vb, nd, sim->c.dt, Fb[0]);
            ADJ_CK(cudaGetLastError());
        }

        for (uint64_t g = n_seg; g-- > 0;) {
            const uint64_t len = std::min<uint64_t>(len_max, n_steps - g * len_max);
            const long long first = (long long)(step0 + g * len_max);
            if (g + 1 < n_seg) {
                ADJ_CK(cudaMemcpyAsync(seg, ckpt + g * nd, state_bytes, cudaMemcpyDeviceToDevice, s));
                ADJ_CK(cudaMemcpyAsync(seg_steps, &first, sizeof(long long), cudaMemcpyHostToDevice, s));
                // the simulation's own step kernel (every CSR kernel gives bit-identical states)
                for (uint64_t k = 0; k < len; ++k)
                    ADJ_CK(titan::enqueue_sim_step_io(sim, s, seg + k * nd, seg + (k + 1) * nd, seg_steps + k,
                                                      seg_steps + k + 1, k > 0));
            }
            for (uint64_t k = len; k-- > 0;) {
                // the clock's phase as titan::clock_phase forms it
                const unsigned long long turns = (unsigned long long)(first + (long long)k) * sim->c.act_turns;
                const double ph = (double)((float)(turns >> 40) * 3.74507028e-7f);
                const float2 sc = make_float2((float)std::sin(ph), (float)std::cos(ph));
                const MassState *X = seg + k * nd;
                auto launch = [&](auto kern) {
                    kern<<<ga, kAdjT, 0, s>>>(X, Fb[cur], Fb[cur ^ 1], xb, vb, nd, sim->d_slice_off, sim->d_adj_nbr,
                                              row, sim->has_c ? sim->d_c : nullptr, sim->c, sc, gacc);
                    return cudaGetLastError();
                };
                if (sim->c.ground) ADJ_CK(sim->has_c ? launch(k_adj_step<true, true>) : launch(k_adj_step<false, true>));
                else ADJ_CK(sim->has_c ? launch(k_adj_step<true, false>) : launch(k_adj_step<false, false>));
                cur ^= 1;
            }
        }
        if (S) {
            k_adj_gather<<<(S + kT - 1) / kT, kT, 0, s>>>(gacc, sim->d_adj_owner, sim->d_kl, sim->d_act, S, grad_amp_dev,
                                                          grad_phase_dev);
            ADJ_CK(cudaGetLastError());
        }
    }
done:
    for (void *p : {(void *)ckpt, (void *)seg, (void *)xb, (void *)vb, (void *)Fb[0], (void *)Fb[1], (void *)seg_steps,
                    (void *)gacc, (void *)row})
        if (p) cudaFreeAsync(p, s);
    if (prev >= 0) cudaSetDevice(prev);
out:
    sim->busy.store(false);
    return st_;
}
