// ne_md.cu -- dynamics kernels of libne.so: the fused lambda-blend + Einstein
// spring + work increment + BAOAB Langevin step, Maxwell-Boltzmann initial
// velocities, the spring energy, and small reductions (msd samples, exported
// energies/forces).
#include <type_traits>

#include "ne_internal.cuh"

namespace {

// ------------------------------------------------------------ fused step
// Total force of H(lambda) on atom i from the EAM force F0, the spring force
// F_E = -k u and, with the centre of mass fixed, their replica means:
//   Frenkel-Ladd (eq. interp): (1 - lambda) F0 + lambda F_E
//   reversible scaling (eq. H_rs): lambda F0
//
// With s the global step and Lambda(s) the schedule:
//   do_close: v += dt/2m F(x_s; Lambda(s))      (second half kick of step s-1)
//   do_open:  W += (Lambda(s+1) - Lambda(s)) dH/dlambda(x_s)   (first thread
//             of the replica; the discrete work sum of Sec. II.A)
//             v += dt/2m F(x_s; Lambda(s+1));  x += dt/2 v;
//             v = c1 v + c2 (xi - mean xi);    x += dt/2 v
// then the tile partials at the resulting x (U_E, sum u, sum |u|^2) and the
// kinetic energy of the completed velocity v_s, the copies of x for
// the pair passes, the
// displacement check against the list-build positions, and the normals of the
// next step with their sums (counter-based, so drawn one step ahead, one
// thread an atom; the prep launch draws the first step's).
//
// With the barostat (RepDev.npt), after the second drift ln V takes one
// Euler-Maruyama step of the overdamped Langevin equation whose stationary
// density is V^(N'+1) exp(-(lambda U + P0 V)/kT) at fixed scaled
// coordinates (N' = dof / 3; the Ito drift includes the derivative of the
// mobility kT m / V, which cancels the Jacobian's kT / V):
//   d ln V = m [(dof kT + lambda W)/(3V) - P0] dt + sqrt(2 kT m dt / V) eta,
// W the virial at x_s (replica totals of pass 2 of this step), eta the first
// normal of Philox stream 5 at (atom 0, step s).  Every block computes the
// same factor and scales its positions about the origin; the replica's last
// block then scales the box.
//
// Per axis (RepDev.npt = 2, for non-cubic cells such as hcp, whose c/a the
// isotropic form cannot change): each eps_a = ln L_a takes the same kind of
// step with the measure dL_x dL_y dL_z,
//   d eps_a = m [(dof/3 kT + lambda W_a)/V - P0] dt + sqrt(2 kT m dt / V) eta_a,
// W_a = -dU/d eps_a the a-th diagonal element of the virial, eta_a the a-th
// normal of the same Philox block; coordinate a and edge a scale by e^(d eps_a).
//
// Lanes 0 .. 2 of a warp take one axis each (z: the axis' normal, drawn before
// the wait for pass 2) and return its factor.  One lane with the normals, two
// divisions, the square root and exp took ~300 FP64 instructions, one every
// ~64 cycles, in every block's way: four bcc 6^3 mixed 33.9 -> 28.5 us a step,
// two bcc 10^3 per axis 41.2 -> 34.2, two bcc 6^3 in FP64 53.8 -> 48.1.  (The step
// kernel as compiled with it: 128 atoms in FP64 without a barostat 25.8 -> 25.4,
// 20 replicas in FP64 273 -> 277.)
__device__ __forceinline__ double npt_scale(const RepDev& P, const double* T, double lam, double z, double dt)
{
    const int a = threadIdx.x & 31;
    const double iv = 1.0 / (P.L[0] * P.L[1] * P.L[2]);
    const double noise = sqrt(2.0 * P.kT * P.mp * dt * iv) * z;
    if (a >= 3) return 1.0;
    double x;
    if (P.npt == 2) {
        x = P.mp * ((P.dof * (1.0 / 3.0) * P.kT + lam * T[TOT_VXX + a]) * iv - P.P0) * dt + noise;
    } else {
        const double W = T[TOT_VXX] + T[TOT_VYY] + T[TOT_VZZ];
        x = (P.mp * ((P.dof * P.kT + lam * W) * (1.0 / 3.0) * iv - P.P0) * dt + noise) * (1.0 / 3.0);
    }
    return 1.0 + ne_baro_expm1(x);
}

// The work increment (lambda_{s+1} - lambda_s) dH/dlambda(x_s) of replica
// rep into W (and its cumulative record and trace row), by one thread.
__device__ void step_work(const DevBatch& B, const Sched& S, const double* T, int rep, long long s, double lam_s,
                          double lam_n)
{
    const double U0 = T[TOT_UEMB] + T[TOT_UPAIR];
    const double g = S.path == 0 ? U0 - T[TOT_UE] : U0;
    const double dW = (lam_n - lam_s) * g;
    int slot = -1;
    long long k = 0;
    if (S.kind == SCHED_FIXED) {
        slot = 0;
    } else if (s >= S.t_eq && s < S.t_eq + S.t_s) {
        slot = 0;
        k = s - S.t_eq;
    } else if (s >= 2 * S.t_eq + S.t_s && s < 2 * S.t_eq + 2 * S.t_s) {
        slot = 1;
        k = s - (2 * S.t_eq + S.t_s);
    }
    if (slot >= 0) {
        double* W = B.W + (S.kind == SCHED_FIXED ? rep : 2 * rep + slot);
        *W += dW;
        if (B.Wcum && S.kind == SCHED_SWITCH) {
            double* wc = B.Wcum + ((size_t)(2 * rep + slot)) * (S.t_s + 1);
            if (k == 0) wc[0] = 0.0;
            wc[k + 1] = *W;
        }
    }
    if (B.trace && s % B.trace_stride == 0 && s / B.trace_stride < B.trace_rows) {
        double* row = B.trace + 8 * (s / B.trace_stride);
        row[0] = (double)s;
        row[1] = lam_s;
        row[2] = g;
        row[3] = U0;
        row[4] = T[TOT_UE];
        row[6] = B.W[2 * rep];
        row[7] = B.W[2 * rep + 1];
        if (slot == 0) row[6] -= dW;
        if (slot == 1) row[7] -= dW;
    }
}

// One thread per atom and component: warp w of a tile's block has component
// w / 2 of 32 atoms.  GB300 issues an FP64 instruction of a warp every ~64
// cycles, so a step's time at small sizes is the number of them in one warp: with
// one thread an atom the FP64 step took 17 us at 128 atoms, now 11 (33 and 34
// at 40,480, where the FP64 Box-Muller, twice the rest, sets it), the mixed one
// 7.7 us at 2000 atoms, now 6.6.
// What every atom of the block shares (lambda, the centre-of-mass means, the
// barostat's factors, the box) is formed once, a lane each, from the schedule's
// table and the replica's totals.  Mixed precision: velocities, kicks and
// thermostat in FP32, each drift added to the FP64 position once, tile sums in
// double-float -- the crystal runner's precision.
constexpr int STEP_THREADS = 3 * NE_TILE;

template <bool MIXED>
__global__ void __launch_bounds__(STEP_THREADS)
    k_step(DevBatch B, Sched S, const long long* __restrict__ step_base, int j, int do_close, int do_open)
{
    using R = typename std::conditional<MIXED, float, double>::type;
    __shared__ double s_lam[2], s_mu[3], s_L[3];
    __shared__ R s_mean[9];             // mean F0, spring and noise terms (see below)
    __shared__ float s_Lf[3], s_iLf[3]; // box and 1 / box after this step's scaling
    __shared__ R s_tab[4][NE_MAX_SPECIES_DEV + 1];  // m, k, c2, dt / 2m: species 0.., the replica's last
    __shared__ float s_w[3][NE_TILE], s_d2[3][NE_TILE];
    __shared__ int s_code[3][NE_TILE];
    __shared__ double s_x64[MIXED ? 1 : 3][NE_TILE];
    __shared__ double s_red[MIXED ? 1 : 5][3][NE_TILE + 1];
    __shared__ float2 s_dff[MIXED ? 5 : 1][6];
    const int tile = blockIdx.x;
    const int rep = B.tile_rep[tile];
    const RepDev& P = B.rep[rep];
    const int c = threadIdx.x / NE_TILE, al = threadIdx.x % NE_TILE;  // component (warp-uniform), atom of the tile
    const int a = (tile - P.tile0) * NE_TILE + al;
    const bool valid = a < P.n;
    const size_t e = 3 * (size_t)(P.off + (valid ? a : 0)) + c;
    const long long s = __ldcg(step_base) + j;  // from L2: the last chunk's end advanced it
    const double* T = B.tot + (size_t)rep * NTOT;
    const bool draw = do_open || !do_close;  // a step follows: its normals
    const bool prep = !do_open && !do_close;
    // the normals of the coming step, which depend on nothing that a kernel of
    // the chain writes, while pass 2 drains
    R z = 0;
    if (valid && draw) {
        const uint4 ph = ne_philox_block(P.seed, P.replica, (unsigned)S.stream, (unsigned)a,
                                         (unsigned long long)(do_open ? s + 1 : s));
        z = MIXED ? (R)ne_normal32(ph, c) : (R)ne_normal64(ph, c);
    }
    double zb = 0.0;  // the barostat's, by lanes 0 .. 2
    if (do_open && P.npt && threadIdx.x < 3)
        zb = ne_normal64(ne_philox_block(P.seed, P.replica, (unsigned)STREAM_BARO, 0u, (unsigned long long)s),
                         P.npt == 2 ? threadIdx.x : 0);
    ne_chain();
    if (threadIdx.x < 32) {
        // lanes 0-8: mean F0, the spring's mean and the noise mean (per unit
        // mass with species tables: the mass-weighted constraint); 9-11 the
        // box after the barostat's step; 12, 13 lambda at s and s + 1
        const int l = threadIdx.x, d = l % 3;
        const double* lam = B.lam + (s - B.lam_s0);
        const double muc = do_open && P.npt ? __shfl_sync(0xffffffffu, npt_scale(P, T, lam[1], zb, S.dt), d) : 1.0;
        if (l < 9) {
            double v = T[l < 3 ? TOT_F0X + d : (l < 6 ? TOT_UX + d : TOT_XIX + d)];
            if (l >= 3 && l < 6) v *= P.nsp ? -1.0 : -P.k;
            s_mean[l] = S.fix_cm ? (R)(v * P.inv_w) : (R)0;
        } else if (l < 12) {
            const double L = P.npt ? muc * P.L[d] : P.L[d];
            s_mu[d] = muc;
            s_L[d] = L;
            s_Lf[d] = P.npt ? (float)L : P.Lf[d];
            s_iLf[d] = P.npt ? 1.f / (float)L : P.iLf[d];
        } else if (l < 14) {
            s_lam[l - 12] = lam[l - 12];
        }
    } else if (threadIdx.x < 33 + NE_MAX_SPECIES_DEV) {
        const int t = threadIdx.x - 32;
        const bool r1 = t == NE_MAX_SPECIES_DEV;  // the replica's single-species values
        const int ts = r1 ? 0 : t;
        if (r1 || t < P.nsp) {
            s_tab[0][t] = (R)(r1 ? P.m : P.ms[ts]);
            s_tab[1][t] = (R)(r1 ? P.k : P.ks[ts]);
            s_tab[2][t] = (R)(r1 ? P.c2 : P.c2s[ts]);
            s_tab[3][t] = (R)(r1 ? P.hdt_m : P.hdts[ts]);
        }
    }
    // this component's state, while the shared values form
    double x = 0.0, x0 = 0.0, vd = 0.0;
    R F0 = 0, xi = 0;
    int q = NE_MAX_SPECIES_DEV;
    float pb = 0.f;
    if (valid) {
        x = B.x[e];
        vd = B.v[e];
        x0 = B.x0[e];
        if (do_close || do_open) F0 = MIXED ? (R)((const float*)B.f32)[4 * (size_t)(P.off + a) + c] : (R)B.f64[e];
        if (do_open) xi = MIXED ? (R)B.xi32[e] : (R)B.xi64[e];
        if (P.nsp) q = P.sp[a];
        pb = ((const float*)B.pbuild)[4 * (size_t)(P.off + a) + c];
    }
    __syncthreads();
    const R ls = (R)s_lam[0], ln = (R)s_lam[1];
    const R mi = s_tab[0][q], ki = s_tab[1][q], c2i = s_tab[2][q], hdti = s_tab[3][q];
    R v = (R)vd, p_ke = 0, p_ux = 0, p_u2 = 0, p_xi = 0;
    int bad = 0;
    if (valid) {
        R u = (R)(x - x0);
        // with species tables F_i -= m_i sum_j F_j / M
        const R wm = P.nsp ? mi : (R)1;
        const R f0 = F0 - wm * s_mean[c], fe = -ki * u - wm * s_mean[3 + c];
        const auto blend = [&](R lam) { return S.path == 0 ? ((R)1 - lam) * f0 + lam * fe : lam * f0; };
        if (do_close) v += hdti * blend(ls);
        if (B.trace) p_ke = (R)0.5 * mi * v * v;
        if (do_open) {
            // velocity increments of the thermostat: c2 (xi - mean xi) for one
            // species; c2_i xi_i - sum_j m_j c2_j xi_j / M with species tables
            const R dv = P.nsp ? c2i * xi - s_mean[6 + c] : c2i * (xi - s_mean[6 + c]);
            v += hdti * blend(ln);
            const R v1 = v;
            v = (MIXED ? (R)P.c1f : (R)P.c1) * v + dv;
            if constexpr (MIXED) {
                const float dx = S.hdtf * (v1 + v);
                if (!isfinite(dx)) bad |= ST_ENAN;
                x += (double)dx;
            } else {
                x = fma(0.5 * S.dt, v1, x);
                x = fma(0.5 * S.dt, v, x);
            }
            if (P.npt) x *= s_mu[c];
            // from x itself, so that a run resumed from (x, v) forms the same totals
            u = (R)(x - x0);
            B.x[e] = x;
        }
        if (!isfinite(x) || !isfinite(v)) bad |= ST_ENAN;
        if (do_close || do_open) B.v[e] = (double)v;
        p_ux = P.nsp ? ki * u : u;
        p_u2 = u * u;
        // x wrapped, its image against the list build's and the displacement from
        // there
        double xw = x;
        float w;
        ne_wrap(xw, w, s_L[c], s_iLf[c]);
        if constexpr (!MIXED) s_x64[c][al] = xw;
        const float nb = rintf((w - pb) * s_iLf[c]), d = fmaf(-s_Lf[c], nb, w - pb);
        // (a position that no wrap takes into the box: no image code, but a list
        // built around it)
        const bool in = fabsf(nb) <= 1.f;
        s_w[c][al] = w;
        s_d2[c][al] = in || isnan(nb) ? d * d : __int_as_float(0x7f800000);
        s_code[c][al] = in ? (int)nb : 0;
        if (draw) {
            if constexpr (MIXED) B.xi32[e] = z;
            else B.xi64[e] = z;
            p_xi = P.nsp ? mi * c2i * z : z;
        }
    }
    if (bad) ne_set_status(B.status, bad);
    // the list of the sites is built: the first step's list kernel has nothing
    // to do (pass 1 clears the mark of a build inside the run)
    if (prep && threadIdx.x == 0 && tile == P.tile0) B.building[rep] = 0;
    if (do_open && threadIdx.x == STEP_THREADS - 32 && tile == P.tile0)
        step_work(B, S, T, rep, s, s_lam[0], s_lam[1]);
    // the tile's partials: UX.. and the normals per component, U2, U_E and KE
    // over the components.  Mixed: double-float, a fixed tree in each warp, then
    // the warps in order; FP64: rows of 64 in shared memory, eight threads a row
    const R p_ue = P.nsp ? (R)0.5 * ki * p_u2 : (R)0;  // one species: U_E is k/2 times the sum of u^2
    const int nq = P.nsp || B.trace ? 5 : 3;
    const R pq[5] = {p_ux, p_u2, p_xi, p_ue, p_ke};
    if constexpr (MIXED) {
        const int wp = threadIdx.x >> 5;
#pragma unroll
        for (int k = 0; k < 5; ++k)
            if (k < nq) {
                const dff t = dff_warp_sum({pq[k], 0.f});
                if ((threadIdx.x & 31) == 0) s_dff[k][wp] = make_float2(t.hi, t.lo);
            }
    } else {
#pragma unroll
        for (int k = 0; k < 5; ++k)
            if (k < nq) s_red[k][c][al] = pq[k];
    }
    __syncthreads();
    double* const pbt = B.partB + tile;
    const size_t np = B.n_tiles;
    if constexpr (MIXED) {
        if (threadIdx.x < 15 && threadIdx.x / 3 < nq) {
            const int k = threadIdx.x / 3, d = threadIdx.x % 3;
            float2* const pf = (float2*)B.partB + tile;
            dff t = dff_add({s_dff[k][2 * d].x, s_dff[k][2 * d].y}, {s_dff[k][2 * d + 1].x, s_dff[k][2 * d + 1].y});
            if (k == 0 || k == 2) {
                pf[((k == 0 ? PB_UX : PB_XIX) + d) * np] = make_float2(t.hi, t.lo);
            } else if (d == 0 && (k != 3 || P.nsp)) {
                for (int w2 = 2; w2 < 6; ++w2) t = dff_add(t, {s_dff[k][w2].x, s_dff[k][w2].y});
                pf[(k == 1 ? PB_U2 : (k == 3 ? PB_UE : PB_KE)) * np] = make_float2(t.hi, t.lo);
                if (k == 1 && !P.nsp) {
                    const double ue = 0.5 * P.k * ((double)t.hi + (double)t.lo);
                    const float h = (float)ue;
                    pf[PB_UE * np] = make_float2(h, (float)(ue - (double)h));
                }
            }
        }
    } else if (threadIdx.x < 128) {
        const int row = threadIdx.x >> 3, sg = threadIdx.x & 7, k = row / 3, d = row % 3;
        const bool on = k < nq;
        const double* r = s_red[on ? k : 0][d] + sg * 8;
        double t = r[0];
#pragma unroll
        for (int z = 1; z < 8; ++z) t += r[z];
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
        if (on && sg == 0) {
            if (k == 0 || k == 2) pbt[((k == 0 ? PB_UX : PB_XIX) + d) * np] = t;
            else s_red[k][d][NE_TILE] = t;  // the pad column
        }
    }
    // the atom's copies for the pair passes, from its three components
    if (threadIdx.x < NE_TILE && valid) {
        const int i = P.off + a;
        B.pos32[i] = make_float4(s_w[0][al], s_w[1][al], s_w[2][al],
                                 __int_as_float(9 * s_code[0][al] + 3 * s_code[1][al] + s_code[2][al]));
        if constexpr (!MIXED) B.pos64[i] = ned4{s_x64[0][al], s_x64[1][al], s_x64[2][al], 0.0};
        if (s_d2[0][al] + s_d2[1][al] + s_d2[2][al] > P.half_skin2) B.flags[rep] = 1;
    }
    if constexpr (!MIXED) {
        __syncthreads();
        // U2; U_E with species tables; KE with a trace
        if (threadIdx.x == 0 || (threadIdx.x == 1 && P.nsp) || (threadIdx.x == 2 && nq == 5)) {
            const int k = threadIdx.x == 0 ? 1 : 2 + threadIdx.x;
            const double t = s_red[k][0][NE_TILE] + s_red[k][1][NE_TILE] + s_red[k][2][NE_TILE];
            pbt[(k == 1 ? PB_U2 : (k == 3 ? PB_UE : PB_KE)) * np] = t;
            if (k == 1 && !P.nsp) pbt[PB_UE * np] = 0.5 * P.k * t;
        }
    }
    // the box of a barostatted replica, by its last block (every block has
    // read the box).  A box whose cells became shorter than r_c + skin, or whose
    // edge fell below 2 (r_c + skin), is reported (NE_ERANGE) and left unchanged.
    if (do_open && P.npt && threadIdx.x == 0) {
        __threadfence();
        if (atomicAdd(&B.tile_done[rep], 1u) == (unsigned)P.ntile - 1u) {
            __threadfence();
            B.tile_done[rep] = 0u;
            RepDev& Pw = const_cast<RepDev*>(B.rep)[rep];
            const double rl = sqrt(P.rlist2);
            bool ok = true;
            for (int d = 0; d < 3; ++d)
                ok = ok && s_L[d] > 2.0 * rl && (P.nc[d] == 0 || s_L[d] / P.nc[d] >= rl);
            if (!ok) ne_set_status(B.status, ST_ERANGE);
            else
                for (int d = 0; d < 3; ++d) {
                    Pw.L[d] = s_L[d];
                    Pw.invL[d] = 1.0 / s_L[d];
                    Pw.Lf[d] = (float)Pw.L[d];
                    Pw.iLf[d] = (float)Pw.invL[d];
                }
        }
    }
}

// Trace temperature column: KE of v_s (tile partials of the step kernel of
// step s) summed in fixed order after that kernel.
__global__ void k_trace_T(DevBatch B, const long long* __restrict__ step_base, int j)
{
    const long long s = *step_base + j;
    if (!B.trace || s % B.trace_stride != 0 || s / B.trace_stride >= B.trace_rows) return;
    const RepDev& P = B.rep[0];
    const double ke = ne_warp_part_sum(B, B.partB, (size_t)PB_KE * B.n_tiles + P.tile0, P.ntile);
    const double kB = 8.617333262e-5;
    if (threadIdx.x == 0) B.trace[8 * (s / B.trace_stride) + 5] = 2.0 * ke / (P.dof * kB);
}

__global__ void k_advance(long long* step_base, long long by) { *step_base += by; }

__global__ void k_set_step(long long* step_base, long long s) { *step_base = s; }

// The replicas' table, tile map and cleared words of a batch, SETUP_REPS replicas
// a launch: the table travels as the kernel's argument, one launch instead of two
// copies from pageable memory and four clears (the FP32 energy of 128 atoms, a
// call and its outputs: 130 -> 122 us; with the status word read by a copy, too).
struct SetupArgs {
    RepDev r[ne::SETUP_REPS];
    int r0;
};
static_assert(sizeof(SetupArgs) <= 4000, "a launch's arguments");

__global__ void __launch_bounds__(128) k_setup(const __grid_constant__ SetupArgs A, RepDev* rep, int* tile_rep,
                                               unsigned* tile_done, int* flags, int* status, double* tot)
{
    const int r = A.r0 + blockIdx.x, t = threadIdx.x;
    const int* src = (const int*)&A.r[blockIdx.x];
    for (int q = t; q < (int)(sizeof(RepDev) / sizeof(int)); q += blockDim.x) ((int*)(rep + r))[q] = src[q];
    for (int q = t; q < A.r[blockIdx.x].ntile; q += blockDim.x) tile_rep[A.r[blockIdx.x].tile0 + q] = r;
    if (t < NTOT) tot[(size_t)r * NTOT + t] = 0.0;
    if (t == 0) {
        tile_done[r] = 0u;
        flags[r] = 0;
        if (r == 0) *status = 0;
    }
}

__global__ void k_status_out(const int* status, int* host)
{
    ne_chain();
    *host = *status;
}

__global__ void k_noise(unsigned long long seed, unsigned replica, int stream, long long step, int n,
                        int mixed, double* z)
{
    for (int a = blockIdx.x * blockDim.x + threadIdx.x; a < n; a += gridDim.x * blockDim.x) {
        uint4 w = ne_philox_block(seed, replica, (unsigned)stream, (unsigned)a, (unsigned long long)step);
        if (mixed) {
            float f[3];
            ne_normals32(w, f);
            for (int c = 0; c < 3; ++c) z[3 * a + c] = f[c];
        } else {
            double d[3];
            ne_normals64(w, d);
            for (int c = 0; c < 3; ++c) z[3 * a + c] = d[c];
        }
    }
}

// ------------------------------------------------------------ velocities
// Philox normals (stream 1, step 0) times sqrt(kT/m); mean removed when the
// centre of mass is fixed; rescaled to exactly T over the free dof.
// Velocity start: Maxwell-Boltzmann from Philox normals, the centre-of-mass
// momentum removed, then scaled to T exactly.  Three launches over the
// tiles (draw, centre, scale); each block forms its replica's sums from the
// tile partials in a fixed order (the partA slots of pass 1 and 2, which a
// force evaluation rewrites before it reads them), so the FP64 Box-Muller of
// a large replica spreads over the SMs instead of one block doing it all.
__device__ __forceinline__ double tile_sum64(double v, double* red)
{
    red[threadIdx.x] = v;
    __syncthreads();
    for (int w = NE_TILE / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    const double t = red[0];
    __syncthreads();
    return t;
}

__device__ __forceinline__ double init_mass(const RepDev& P, int a) { return P.nsp ? P.ms[P.sp[a]] : P.m; }

__global__ void __launch_bounds__(NE_TILE) k_init_v_draw(DevBatch B)
{
    __shared__ double red[NE_TILE];
    const int tile = blockIdx.x;
    const RepDev& P = B.rep[B.tile_rep[tile]];
    const int a = (tile - P.tile0) * NE_TILE + threadIdx.x;
    // with species tables atom a has sd = sqrt(kT / m_a), and the momentum
    // sum_a m_a v_a / M is removed (the mass-weighted centre of mass)
    double sum[3] = {0, 0, 0};
    if (a < P.n) {
        const double sd = sqrt(P.kT / init_mass(P, a));
        const double w = P.nsp ? init_mass(P, a) / P.M : 1.0;
        double z[3];
        ne_normals64(ne_philox_block(P.seed, P.replica, STREAM_INITV, (unsigned)a, 0ull), z);
        for (int c = 0; c < 3; ++c) {
            B.v[3 * (P.off + a) + c] = sd * z[c];
            sum[c] = w * sd * z[c];
        }
    }
    for (int c = 0; c < 3; ++c) {
        const double t = tile_sum64(sum[c], red);
        if (threadIdx.x == 0) B.partA[(size_t)c * B.n_tiles + tile] = t;
    }
}

__global__ void __launch_bounds__(NE_TILE) k_init_v_center(DevBatch B, int fix_cm)
{
    __shared__ double red[NE_TILE];
    __shared__ double s_mean[3];
    const int tile = blockIdx.x;
    const RepDev& P = B.rep[B.tile_rep[tile]];
    if (threadIdx.x < 32)
        for (int c = 0; c < 3; ++c) {
            const double t = ne_warp_part_sum(B.partA + (size_t)c * B.n_tiles + P.tile0, P.ntile);
            if (threadIdx.x == 0) s_mean[c] = fix_cm ? (P.nsp ? t : t / P.n) : 0.0;
        }
    __syncthreads();
    const int a = (tile - P.tile0) * NE_TILE + threadIdx.x;
    double ke = 0.0;
    if (a < P.n)
        for (int c = 0; c < 3; ++c) {
            double* vv = &B.v[3 * (P.off + a) + c];
            *vv -= s_mean[c];
            ke += 0.5 * init_mass(P, a) * (*vv) * (*vv);
        }
    const double t = tile_sum64(ke, red);
    if (threadIdx.x == 0) B.partA[(size_t)3 * B.n_tiles + tile] = t;
}

__global__ void __launch_bounds__(NE_TILE) k_init_v_scale(DevBatch B)
{
    __shared__ double s_sc;
    const int tile = blockIdx.x;
    const RepDev& P = B.rep[B.tile_rep[tile]];
    if (threadIdx.x < 32) {
        const double ke = ne_warp_part_sum(B.partA + (size_t)3 * B.n_tiles + P.tile0, P.ntile);
        const double kB = 8.617333262e-5;
        if (threadIdx.x == 0) s_sc = sqrt((P.kT / kB) / (2.0 * ke / (P.dof * kB)));
    }
    __syncthreads();
    const int a = (tile - P.tile0) * NE_TILE + threadIdx.x;
    if (a < P.n)
        for (int c = 0; c < 3; ++c) B.v[3 * (P.off + a) + c] *= s_sc;
}

// ------------------------------------------------------------ spring
// Einstein crystal (eq. einstein): U_E = sum k/2 |r - r0|^2, F_E = -k (r - r0).
__global__ void __launch_bounds__(1024) k_spring(const double* __restrict__ x, const double* __restrict__ x0,
                                                 int n, double k, double* f, double* e)
{
    __shared__ double red[1024];
    double acc = 0.0;
    for (int q = threadIdx.x; q < 3 * n; q += blockDim.x) {
        double u = x[q] - x0[q];
        acc += 0.5 * k * u * u;
        if (f) f[q] = -k * u;
    }
    red[threadIdx.x] = acc;
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w) red[threadIdx.x] += red[threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x == 0 && e) *e = red[0];
}

// EAM forces, times scale, and energy of replica 0 to caller buffers.
template <bool MIXED>
__global__ void k_export(DevBatch B, double* f, double* e, double scale)
{
    ne_chain();
    const RepDev& P = B.rep[0];
    if (f)
        for (int q = blockIdx.x * blockDim.x + threadIdx.x; q < 3 * P.n; q += gridDim.x * blockDim.x) {
            const size_t i = (size_t)P.off + q / 3;
            f[q] = scale * (MIXED ? (double)((const float*)B.f32)[4 * i + q % 3] : B.f64[3 * i + q % 3]);
        }
    if (blockIdx.x == 0 && threadIdx.x == 0 && e) *e = B.tot[TOT_UEMB] + B.tot[TOT_UPAIR];
}

// One msd sample per replica from the step-kernel partials:
// (1/n) sum |u_i - mean u|^2 = (1/n) sum |u|^2 - |mean u|^2.
__global__ void k_msd_sample(DevBatch B, double* acc)
{
    const int rep = blockIdx.x;
    const RepDev& P = B.rep[rep];
    double s[4];
    s[0] = ne_warp_part_sum(B, B.partB, (size_t)PB_UX * B.n_tiles + P.tile0, P.ntile);
    s[1] = ne_warp_part_sum(B, B.partB, (size_t)PB_UY * B.n_tiles + P.tile0, P.ntile);
    s[2] = ne_warp_part_sum(B, B.partB, (size_t)PB_UZ * B.n_tiles + P.tile0, P.ntile);
    s[3] = ne_warp_part_sum(B, B.partB, (size_t)PB_U2 * B.n_tiles + P.tile0, P.ntile);
    if (threadIdx.x != 0) return;
    const double invN = 1.0 / P.n;
    acc[rep] += s[3] * invN - (s[0] * s[0] + s[1] * s[1] + s[2] * s[2]) * invN * invN;
}

// One msd sample per species of each replica with species tables (Sec. V):
// displacements u_i = x_i - x0_i taken about the mass-weighted centre,
// dR = sum_i m_i u_i / M; acc[rep * NE_MAX_SPECIES + s] += (1/N_s) sum over
// the atoms of species s of |u_i - dR|^2.  One block per replica, FP64,
// fixed-order block sums.
__global__ void __launch_bounds__(256) k_msd_sample_species(DevBatch B, double* acc)
{
    __shared__ double red[3 + 2 * NE_MAX_SPECIES_DEV][256];
    const int rep = blockIdx.x;
    const RepDev& P = B.rep[rep];
    double s[3] = {0, 0, 0};
    for (int a = threadIdx.x; a < P.n; a += blockDim.x) {
        const double w = P.ms[P.sp[a]] / P.M;
        for (int c = 0; c < 3; ++c) s[c] += w * (B.x[3 * (P.off + a) + c] - B.x0[3 * (P.off + a) + c]);
    }
    for (int c = 0; c < 3; ++c) red[c][threadIdx.x] = s[c];
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w)
            for (int c = 0; c < 3; ++c) red[c][threadIdx.x] += red[c][threadIdx.x + w];
        __syncthreads();
    }
    const double dR[3] = {red[0][0], red[1][0], red[2][0]};
    __syncthreads();
    double d2[NE_MAX_SPECIES_DEV] = {}, cnt[NE_MAX_SPECIES_DEV] = {};
    for (int a = threadIdx.x; a < P.n; a += blockDim.x) {
        const int q = P.sp[a];
        for (int c = 0; c < 3; ++c) {
            const double d = (B.x[3 * (P.off + a) + c] - B.x0[3 * (P.off + a) + c]) - dR[c];
            d2[q] += d * d;
        }
        cnt[q] += 1.0;
    }
    for (int q = 0; q < NE_MAX_SPECIES_DEV; ++q) {
        red[3 + q][threadIdx.x] = d2[q];
        red[3 + NE_MAX_SPECIES_DEV + q][threadIdx.x] = cnt[q];
    }
    __syncthreads();
    for (int w = blockDim.x / 2; w > 0; w >>= 1) {
        if (threadIdx.x < w)
            for (int q = 3; q < 3 + 2 * NE_MAX_SPECIES_DEV; ++q) red[q][threadIdx.x] += red[q][threadIdx.x + w];
        __syncthreads();
    }
    if (threadIdx.x < P.nsp && red[3 + NE_MAX_SPECIES_DEV + threadIdx.x][0] > 0)
        acc[rep * NE_MAX_SPECIES_DEV + threadIdx.x] +=
            red[3 + threadIdx.x][0] / red[3 + NE_MAX_SPECIES_DEV + threadIdx.x][0];
}

}  // namespace

namespace ne {

void launch_step(const DevBatch& B, const Sched& S, bool mixed, const long long* step_base, int j,
                 int do_close, int do_open, cudaStream_t st)
{
    if (mixed)
        ne_launch(k_step<true>, B.n_tiles, STEP_THREADS, 0, st, B, S, step_base, j, do_close, do_open);
    else
        ne_launch(k_step<false>, B.n_tiles, STEP_THREADS, 0, st, B, S, step_base, j, do_close, do_open);
    if (B.trace && do_open) k_trace_T<<<1, 32, 0, st>>>(B, step_base, j);
}

void launch_noise(unsigned long long seed, unsigned replica, int stream, long long step, int n, int mixed,
                  double* z, cudaStream_t st)
{
    k_noise<<<(n + 255) / 256 < 1024 ? (n + 255) / 256 : 1024, 256, 0, st>>>(seed, replica, stream, step, n,
                                                                            mixed, z);
}

void launch_advance(long long* step_base, long long by, cudaStream_t st)
{
    k_advance<<<1, 1, 0, st>>>(step_base, by);
}

void launch_set_step(long long* step_base, long long s, cudaStream_t st) { k_set_step<<<1, 1, 0, st>>>(step_base, s); }

void launch_setup(const RepDev* reps, int n_rep, RepDev* rep, int* tile_rep, unsigned* tile_done, int* flags,
                  int* status, double* tot, cudaStream_t st)
{
    SetupArgs A;
    for (int r0 = 0; r0 < n_rep; r0 += SETUP_REPS) {
        const int k = n_rep - r0 < SETUP_REPS ? n_rep - r0 : SETUP_REPS;
        for (int q = 0; q < k; ++q) A.r[q] = reps[r0 + q];
        A.r0 = r0;
        k_setup<<<k, 128, 0, st>>>(A, rep, tile_rep, tile_done, flags, status, tot);
    }
}

cudaError_t launch_status_out(const int* status, int* host, cudaStream_t st)
{
    return ne_launch(k_status_out, 1, 1, 0, st, status, host);
}

void launch_init_velocities(const DevBatch& B, int fix_cm, cudaStream_t st)
{
    k_init_v_draw<<<B.n_tiles, NE_TILE, 0, st>>>(B);
    k_init_v_center<<<B.n_tiles, NE_TILE, 0, st>>>(B, fix_cm);
    k_init_v_scale<<<B.n_tiles, NE_TILE, 0, st>>>(B);
}

void launch_spring(const double* x, const double* x0, int n, double k, double* f, double* e,
                   double*, cudaStream_t st)
{
    k_spring<<<1, 1024, 0, st>>>(x, x0, n, k, f, e);
}

void launch_export(const DevBatch& B, bool mixed, double* f_out, double* e_out, double scale, cudaStream_t st)
{
    const int want = f_out ? (3 * B.n_tot + 255) / 256 : 1, grid = want < 4 * B.sms ? want : 4 * B.sms;
    if (mixed)
        ne_launch(k_export<true>, grid, 256, 0, st, B, f_out, e_out, scale);
    else
        ne_launch(k_export<false>, grid, 256, 0, st, B, f_out, e_out, scale);
}

void launch_msd_sample(const DevBatch& B, double* acc, cudaStream_t st)
{
    if (B.species_any)
        k_msd_sample_species<<<B.n_rep, 256, 0, st>>>(B, acc);
    else
        k_msd_sample<<<B.n_rep, 32, 0, st>>>(B, acc);
}

}  // namespace ne
