// ne_cluster.cuh -- replica description and launcher of the persistent
// cluster-per-replica runner for crystals (ne_cluster.cu).
#pragma once
#include <cuda_runtime.h>

#include "ne_internal.cuh"

#define NE_STENCIL_MAX 512  // stencil entries per basis site
#define NE_STENCIL_PAD 16   // far entries ending each basis site's stencil (outside any cutoff)

struct XRep {
    double cell[3];       // cell edges (a, a, a; hcp: a, sqrt(3) a, c)
    double basis[4][3];   // basis positions as fractions of the cell edges
    double k;             // spring constant (FP64 for the mean spring force)
    float kf, mf, hdt_mf, c1f, c2f;
    float D;              // largest displacement from a site the stencil covers
    int n, off, nb, nx, ny, nz;
    int st_off, st_cnt;   // stencil of basis b: entries [st_off + b * st_cnt, + st_cnt)
    int st_margin;        // M: cell offsets of the stencil lie in [-M, M]
    unsigned long long seed;
    unsigned replica;
    int widx;             // index of the replica in the caller's arrays (work W)
    // several species (Sec. V): nsp >= 2 -- atom a has species sp[a]
    // (validated on the host) with spring kfs, half-step factor hdts, noise
    // amplitude c2fs and mass mfs of its species; invM = 1 / total mass
    int nsp;
    const unsigned char* sp;
    float invM;
    float kfs[NE_MAX_SPECIES_DEV], hdts[NE_MAX_SPECIES_DEV], c2fs[NE_MAX_SPECIES_DEV], mfs[NE_MAX_SPECIES_DEV];
    int cta0, ncta;       // brick runner: the replica's first CTA in the grid and its CTA count
    // barostat (reversible-scaling path; reading A23): 0 none, 1 isotropic,
    // 2 one equation per box edge; target pressure, mobility beta_T / tau_p,
    // k_B T, degrees of freedom and the box at the call's start
    int npt, dof;
    double P0, mp, kT;
    double box0[3];
};

// Tensor memory as per-thread scratch (both crystal runners): a CTA that is
// alone on its SM takes all NE_TM_COLS columns; a warp reads and writes
// NE_TM_BATCH columns of its own lanes at a time.
#define NE_TM_COLS 512
#define NE_TM_BATCH 8

// N (4 or 8) consecutive TMEM columns of this thread's lane (32x32b shape:
// thread i of the warp is lane i of the warp's quarter).  The load waits for
// its data; the registers pass through the wait so no use moves above it.
template <int N>
__device__ __forceinline__ void ne_tm_st(unsigned taddr, const float (&v)[N])
{
    static_assert(N == 4 || N == 8, "TMEM batches of 4 or 8 columns");
    if constexpr (N == 8)
        asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                     :
                     : "r"(taddr), "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])),
                       "r"(__float_as_uint(v[2])), "r"(__float_as_uint(v[3])), "r"(__float_as_uint(v[4])),
                       "r"(__float_as_uint(v[5])), "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7]))
                     : "memory");
    else
        asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};"
                     :
                     : "r"(taddr), "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])),
                       "r"(__float_as_uint(v[2])), "r"(__float_as_uint(v[3]))
                     : "memory");
}

template <int N>
__device__ __forceinline__ void ne_tm_ld(unsigned taddr, float (&v)[N])
{
    static_assert(N == 4 || N == 8, "TMEM batches of 4 or 8 columns");
    unsigned r[8];
    if constexpr (N == 8) {
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
                       "=r"(r[7])
                     : "r"(taddr)
                     : "memory");
        asm volatile("tcgen05.wait::ld.sync.aligned;"
                     : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]),
                       "+r"(r[7])
                     :
                     : "memory");
    } else {
        asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                     : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                     : "r"(taddr)
                     : "memory");
        asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]) : : "memory");
    }
#pragma unroll
    for (int q = 0; q < N; ++q) v[q] = __uint_as_float(r[q]);
}

// Four columns of 32-bit words (packed integers) of this thread's lane.
__device__ __forceinline__ void ne_tm_st_u4(unsigned taddr, const unsigned (&v)[4])
{
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};"
                 :
                 : "r"(taddr), "r"(v[0]), "r"(v[1]), "r"(v[2]), "r"(v[3])
                 : "memory");
}

__device__ __forceinline__ void ne_tm_ld_u4(unsigned taddr, unsigned (&v)[4])
{
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3])
                 : "r"(taddr)
                 : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;" : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]) : : "memory");
}

// Eight float columns at taddr_f and four word columns at taddr_w, both
// loads in flight before the one wait.
__device__ __forceinline__ void ne_tm_ld_f8u4(unsigned taddr_f, unsigned taddr_w, float (&f)[8], unsigned (&w)[4])
{
    unsigned r[8];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr_f)
                 : "memory");
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3])
                 : "r"(taddr_w)
                 : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(w[0]), "+r"(w[1]), "+r"(w[2]), "+r"(w[3])
                 :
                 : "memory");
#pragma unroll
    for (int q = 0; q < 8; ++q) f[q] = __uint_as_float(r[q]);
}

// The state of the atom a thread owns, NE_TM_STATE columns of its lane: the
// displacement from its site in fixed point (three 64-bit words), velocity and
// the normals of the coming step.  Kept there between integrations it holds no
// registers through the pair passes, which run at the launch bound's cap.
#define NE_TM_STATE 12
struct ne_atom_state {
    long long xr[3];
    float v[3], xi[3];
};

__device__ __forceinline__ void ne_tm_st_state(unsigned taddr, const ne_atom_state& a)
{
    const unsigned w[12] = {(unsigned)a.xr[0], (unsigned)(a.xr[0] >> 32), (unsigned)a.xr[1], (unsigned)(a.xr[1] >> 32),
                            (unsigned)a.xr[2], (unsigned)(a.xr[2] >> 32), __float_as_uint(a.v[0]), __float_as_uint(a.v[1]),
                            __float_as_uint(a.v[2]), __float_as_uint(a.xi[0]), __float_as_uint(a.xi[1]),
                            __float_as_uint(a.xi[2])};
    asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
                 :
                 : "r"(taddr), "r"(w[0]), "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
                 : "memory");
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1, %2, %3, %4};"
                 :
                 : "r"(taddr + 8u), "r"(w[8]), "r"(w[9]), "r"(w[10]), "r"(w[11])
                 : "memory");
}

// (the stores before it have been waited for: tcgen05.wait::st)
__device__ __forceinline__ void ne_tm_ld_state(unsigned taddr, ne_atom_state& a)
{
    unsigned r[8], w[4];
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
                 : "r"(taddr)
                 : "memory");
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0, %1, %2, %3}, [%4];"
                 : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3])
                 : "r"(taddr + 8u)
                 : "memory");
    asm volatile("tcgen05.wait::ld.sync.aligned;"
                 : "+r"(r[0]), "+r"(r[1]), "+r"(r[2]), "+r"(r[3]), "+r"(r[4]), "+r"(r[5]), "+r"(r[6]), "+r"(r[7]),
                   "+r"(w[0]), "+r"(w[1]), "+r"(w[2]), "+r"(w[3])
                 :
                 : "memory");
#pragma unroll
    for (int c = 0; c < 3; ++c) a.xr[c] = (long long)(((unsigned long long)r[2 * c + 1] << 32) | r[2 * c]);
    a.v[0] = __uint_as_float(r[6]);
    a.v[1] = __uint_as_float(r[7]);
    a.v[2] = __uint_as_float(w[0]);
    a.xi[0] = __uint_as_float(w[1]);
    a.xi[1] = __uint_as_float(w[2]);
    a.xi[2] = __uint_as_float(w[3]);
}

// The barostat of the crystal runners (reading A23), one replica a CTA.  GB300
// issues a warp's FP64 instructions ~64 cycles apart, so what one thread did
// between the virial and the integration -- the FP64 normal, square root,
// divisions and exponential, ~300 of them -- held the whole CTA for ~9 us a step.
// Here the normals of 32 steps are drawn at once, a step per lane, and 1 / V and
// the noise amplitude follow from the box as soon as it is known, both by warps
// that own no atom and while the others integrate; what is left behind the
// virial is ~15 FP64 instructions.
struct ne_baro_smem {
    double z[32][3];      // normals of steps s_begin + 32 k .. + 31 (Philox stream 5, atom 0)
    double mu_tot[3];     // box and lattice sites over those of the call's start, per axis
    double em1[3];        // the step's scale factors minus one
    double inv_v, noise;  // 1 / V and sqrt(2 kT m dt / V)
    float muf[3], em1f[3];  // mu_tot and em1 in FP32
    int small;            // every |em1| below 2e-4 (ne_baro_scale)
    int box_ok;           // two periodic images of a site stay more than 2 r_c apart
};

// normals of the 32 steps from s on, a step per lane
__device__ __forceinline__ void ne_baro_draw(ne_baro_smem& b, const XRep& R, long long s)
{
    double z[3];
    ne_normals64(ne_philox_block(R.seed, R.replica, (unsigned)STREAM_BARO, 0u,
                                 (unsigned long long)(s + (threadIdx.x & 31))),
                 z);
    for (int c = 0; c < 3; ++c) b.z[threadIdx.x & 31][c] = z[c];
}

// 1 / V and the noise amplitude of the box mu_tot, by one thread
__device__ __forceinline__ void ne_baro_box(ne_baro_smem& b, const XRep& R, double dt)
{
    const double V = b.mu_tot[0] * R.box0[0] * b.mu_tot[1] * R.box0[1] * b.mu_tot[2] * R.box0[2];
    b.inv_v = 1.0 / V;
    b.noise = sqrt(2.0 * R.kT * R.mp * dt / V);
}

// The step's scale factors from the diagonal virial W (the same in every lane;
// double-float per axis, and so added over the axes: 48 bits of sums that FP32
// pairs leave good to 24), by lanes 0 .. 2 of one warp; i: the step's place in z
__device__ __forceinline__ void ne_baro_step(ne_baro_smem& b, const XRep& R, const dff (&W)[3], double lam, double dt,
                                             double r_c, int i)
{
    const int a = threadIdx.x & 31;
    if (a < 3) {
        double x;
        if (R.npt == 2) {
            const double Wa = (double)(a == 0 ? W[0].hi : (a == 1 ? W[1].hi : W[2].hi)) +
                              (double)(a == 0 ? W[0].lo : (a == 1 ? W[1].lo : W[2].lo));
            const double drive = (R.dof / 3.0 * R.kT + lam * Wa) * b.inv_v - R.P0;
            x = R.mp * drive * dt + b.noise * b.z[i][a];
        } else {  // isotropic; a replica without the barostat has mp = 0
            const dff w = dff_add(dff_add(W[0], W[1]), W[2]);
            const double drive = (R.dof * R.kT + lam * ((double)w.hi + (double)w.lo)) * (1.0 / 3.0) * b.inv_v - R.P0;
            x = (R.mp * drive * dt + b.noise * b.z[i][0]) * (1.0 / 3.0);
        }
        const double e = ne_baro_expm1(x), mu = fma(e, b.mu_tot[a], b.mu_tot[a]);
        b.em1[a] = e;
        b.mu_tot[a] = mu;
        b.muf[a] = (float)mu;
        const bool ok = mu * R.box0[a] > 2.0 * r_c + 1.2;
        b.em1f[a] = (float)e;
        const unsigned all = __ballot_sync(7u, ok), sm = __ballot_sync(7u, fabs(e) < 2e-4);
        if (a == 0) {
            b.box_ok = all == 7u;
            b.small = sm == 7u;
        }
    }
}

// A displacement in fixed point (2^-32 A) scaled by 1 + em1 of axis c: for
// small factors by its change, from the FP32 displacement u (the change's error,
// 2^-23 of |e u| <= 4e-4 A, is below a quarter of the grid; a usual step's
// e ~ 1e-5 leaves a hundredth), else in FP64
__device__ __forceinline__ long long ne_baro_scale(const ne_baro_smem& b, long long xr, float u, int c)
{
    if (b.small) return xr + (long long)__float2int_rn(b.em1f[c] * u * 4294967296.f);
    return __double2ll_rn(fma(b.em1[c], (double)xr, (double)xr));
}

// Warp 0 of the CTA takes all NE_TM_COLS columns (the base address goes to
// *s_slot in shared memory); the caller then makes it visible with
// tcgen05.fence::before_thread_sync, a CTA barrier and
// tcgen05.fence::after_thread_sync.
__device__ __forceinline__ void ne_tm_alloc(unsigned* s_slot)
{
    if (threadIdx.x < 32) {
        __syncwarp();
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :
                     : "r"((unsigned)__cvta_generic_to_shared(s_slot)), "r"(NE_TM_COLS)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
}

// Every thread of the CTA calls this once it is past its last TMEM access:
// warp 0 returns the columns.
__device__ __forceinline__ void ne_tm_free(unsigned base)
{
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    if (threadIdx.x < 32) {
        __syncwarp();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(base), "r"(NE_TM_COLS) : "memory");
    }
}

namespace ne {
size_t cluster_smem_bytes(int n_max, int nb_nst_max, int lut_max, bool npt = false);
int cluster_atoms_per_cta();
int cluster_threads_per_atom();
int cluster_size_for(int n, int nb);           // smallest CTAs per cluster for an n-atom replica
int cluster_atoms_for(int n, int C, int nb);    // atoms per CTA of an n-atom replica on C CTAs
int cluster_max_active(int C, size_t smem);     // co-resident clusters of C CTAs (0 if none or on error)
cudaError_t launch_lambda_table(const Sched& S, long long s_begin, long long count, double* out, cudaStream_t st);
cudaError_t launch_cluster(const XRep* reps, int n_rep, int C, size_t smem, const float4* st_vec,
                           const float* st_dist, double* x, double* v, double* W, int* status, const Sched& S,
                           long long s_begin, long long n_steps, const Tables& tab, unsigned long long* work,
                           int k_lo, double* lam_tab, double* wcum, cudaStream_t st, bool npt = false,
                           double* boxes_out = nullptr);
// Brick runner (ne_brick.cu): replicas larger than a cluster holds, one
// cooperative launch over CTAs that own blocks of cells and exchange u and
// F' through global memory between barriers of the replica's CTAs; with the
// barostat (npt) a third barrier a step carries the CTAs' virial sums.
size_t brick_smem_bytes(int tpa, int nb_nst_max, int lut_max, bool npt = false);
int brick_atoms_per_cta(int tpa);
int brick_max_ctas(int tpa, size_t smem, bool npt = false);  // co-resident CTAs of the launch (0 on error)
#define NE_BAR_STRIDE 32
struct BrickBufs {
    float4* u4;      // [2][N] (u, F'(rho)) of every atom, by step parity
    float* part;     // [2][n_cta][NPART] per-CTA partial sums, by step parity
    float* vir;      // [n_cta][6] per-CTA diagonal virial (hi, lo per axis; barostat only)
    unsigned* bar;   // [replicas][NE_BAR_STRIDE] barrier arrivals, a cache line each
    int* abortf;     // a bounded wait gave up: every CTA leaves
    double* xs;      // [N][3] positions that the call reached, until they are taken over
    float* vs;       // [N][3] velocities
    double* ws;      // [replicas][5] works and box
    unsigned spin_limit;  // polls, each an L2 round trip, after which a wait gives up
};
#define NE_SPIN_LIMIT (1u << 22)  // a few seconds
cudaError_t launch_brick(int tpa, const XRep* reps, int n_rep, const int* cta_rep, int n_cta, size_t smem, const float4* st_vec,
                         const float* st_dist, double* x, double* v, double* W, int* status, const Sched& S,
                         long long s_begin, long long n_steps, const Tables& tab, unsigned long long* work,
                         int k_lo, const double* lam_tab, double* wcum, const BrickBufs& bb, long long n_tot,
                         cudaStream_t st, bool npt = false, double* boxes_out = nullptr);
}  // namespace ne
