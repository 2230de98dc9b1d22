// ne_internal.cuh -- device-side layouts and helpers shared by the kernels of
// libne.so (not part of the public ABI; see include/ne.h).
//
// Data layout in HBM (all replicas of a batch concatenated, atom-major):
//   x, v, x0            double [N][3]   caller-owned, unwrapped positions
//   pbuild              float4 [N]      wrapped positions at the last list build
//   pos32               float4 [N]      FP32 copy of x wrapped into the box; .w (int bits) the code
//                                       9 a + 3 b + c of the box lengths it lies from the image
//                                       nearest pbuild, which the list's images refer to
//   posF                float4 [N]      (x, y, z, F'(rho)) written by pass 1 (mixed)
//   pos64               ned4 [N]        wrapped positions (x, y, z) and F'(rho) (FP64 path)
//   csort               float4 [N]      the same sorted by cell, .w the atom's index in its replica
//   f32 / f64           EAM forces, float4 [N] (mixed) or double [N][3]
//   xi32 / xi64         Langevin normals of the coming step, [N][3]
//   nbr, ncnt           candidate list within r_c + skin: int [N][NE_NMAX] (neighbour and its
//                       image), count [N]
//   sl, gs, scnt        the step's pairs inside r_c: neighbour and its image, and f'(r)/r of
//                       each -- int [N][NE_SMAX] and double [N][NE_SMAX] (FP64), or (int,
//                       float bits) pairs [N][NE_SMAX] in sl, which then is gs's buffer (mixed);
//                       count [N]
//   partA / partB       partial sums of the pair blocks (pass 1 and 2) and of the
//                       step kernel's tiles, quantity-major
//   tot                 per-replica totals formed by the last block of pass 2
// A tile is NE_TILE consecutive atoms of one replica; tiles never straddle
// replicas, and a pair block takes a whole fraction of a tile, so every
// per-replica sum is a fixed-order sum of partials.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <cmath>

// 32-byte aligned quadruple of doubles (one spline interval in FP64)
struct __align__(32) ned4 {
    double x, y, z, w;
};

#define NE_TILE 64
#define GROUP_TILES 64  // tiles of a replica whose partials pass 2 sums first
#define NE_PAIR_SUB 8   // most pair blocks per tile (32 lanes per atom)
// list entry: neighbour in the low 27 bits, above them the code 9 (a + 1) + 3 (b + 1) + c + 1 of the
// shift (a, b, c), each in {-1, 0, 1}, in box lengths, that is added to r_j - r_i
#define NE_IMG_SHIFT 27
#define NE_IMG_NONE 13
#define NE_MAX_SPECIES_DEV 8  // species per replica (NE_MAX_SPECIES of the public header)
#define NE_NMAX 256   // candidate neighbours per atom (r < r_c + skin)
#define NE_SMAX 128   // neighbours per atom inside r_c
#define NE_RMIN 0.2   // A: shorter pair distances are reported as NE_ERANGE (atoms may overlap at lambda -> 1)

// device status bits
enum { ST_ERANGE = 1, ST_ENEIGH = 2, ST_ENAN = 4, ST_ETIMEOUT = 8, ST_EINVAL = 16 };

// Philox stream ids (low 4 bits of the 4th counter word)
enum { STREAM_FL = 0, STREAM_INITV = 1, STREAM_RS = 2, STREAM_MSD = 3, STREAM_STEP = 4, STREAM_BARO = 5 };

// partials of pass 1 (energies, the pair part of the virial) and pass 2 (forces, its embedding part), at x_k
enum { PA_UEMB = 0, PA_UPAIR, PA_F0X, PA_F0Y, PA_F0Z, PA_VXX, PA_VYY, PA_VZZ, PA_WXX, PA_WYY, PA_WZZ, NPA };
// tile partials of the step kernel (at x_{k+1}; KE of the completed velocity; the normals of step k+1)
enum { PB_UE = 0, PB_UX, PB_UY, PB_UZ, PB_U2, PB_KE, PB_XIX, PB_XIY, PB_XIZ, NPB };
// per-replica totals
enum { TOT_UEMB = 0, TOT_UPAIR, TOT_F0X, TOT_F0Y, TOT_F0Z, TOT_VXX, TOT_VYY, TOT_VZZ, TOT_UE, TOT_UX, TOT_UY, TOT_UZ,
       TOT_XIX, TOT_XIY, TOT_XIZ, NTOT };

struct RepDev {
    double L[3], invL[3];
    float Lf[3], iLf[3];  // the same in FP32 (a conversion costs an FP64 slot)
    double k;        // Einstein spring
    float c1f;       // c1 in FP32
    double c1, c2;   // Ornstein-Uhlenbeck coefficients
    double hdt_m;    // dt / (2 m)
    double kT;
    double m;
    double rlist2;   // (r_c + skin)^2
    float half_skin2;
    int off, n, tile0, ntile;
    int grp0;        // first of its groups of GROUP_TILES tiles
    int nc[3];       // cells per axis; 0 = all pairs
    int bin64;       // cells found in FP64 (see ne_bin64)
    int cell_off;
    int dof;
    unsigned long long seed;
    unsigned replica;
    int npt;         // barostat (RS path): 1 isotropic, 2 one equation per box edge
    double P0, mp;   // target pressure, mobility beta_T / tau_p
    // Several species (Sec. V): nsp = 0 -- every atom has m and k above;
    // nsp >= 2 -- atom a has species sp[a] (validated on the host) with mass
    // ms, spring ks, noise amplitude c2s and half-step factor hdts of its
    // species; M is the replica's total mass.  With species tables the
    // step kernel's sum PB_UX.. holds sum_j k_j u_j and its PB_XIX.. holds
    // sum_j m_j c2_j xi_j: the sums the mass-weighted centre-of-mass
    // constraint needs.
    int nsp;
    const unsigned char* sp;
    double M;
    double inv_w;    // 1 / n, or 1 / M with species tables
    double ms[NE_MAX_SPECIES_DEV], ks[NE_MAX_SPECIES_DEV], c2s[NE_MAX_SPECIES_DEV], hdts[NE_MAX_SPECIES_DEV];
};

// The list build finds a position's cell in FP32, to 3e-7 of the box edge, which
// cells of an edge above r_c + skin + 1e-3 A have room for up to 2000 A.  A replica
// with smaller cells (down to r_c + skin, where an edge is a near multiple of it or
// a barostat contracts the box) or a longer edge has its atoms binned in FP64.
inline void ne_bin64(RepDev& R, double rl)
{
    R.bin64 = R.npt != 0;
    for (int d = 0; d < 3; ++d) R.bin64 |= R.nc[d] > 0 && (R.L[d] < (rl + 1e-3) * R.nc[d] || R.L[d] > 2000.0);
}

// Schedule of a run, shared by the replicas of one launch.
enum { SCHED_SWITCH = 0, SCHED_FIXED = 1 };
struct Sched {
    long long t_eq, t_s;
    double lambda_f;
    double lam_a, lam_b;   // SCHED_FIXED: lambda before / after the jump
    long long s0;          // SCHED_FIXED: step of the jump
    double dt;
    float hdtf;            // dt / 2 in FP32
    int kind, path, fn, stream, fix_cm;
};

struct Tables {
    // phi and f interleaved per interval: [nk-1][2] (phi, f), cubic in u
    const float4* pf32;
    const ned4* pf64;
    const float4* F32;     // embedding, [nk-1]
    const ned4* F64;
    int nk;
    double h_r, inv_h_r, h_rho, inv_h_rho;
    double ih_hi, ih_k, ih_c;  // 1 / h_r = ih_hi (1 + ih_k), ih_hi of 29 bits; (1 + ih_k) / 2
    double r_c, rho_max;
    float inv_h_rf, rcf, rc2f, rmin2f, inv_h_rhof;
    float rho_maxf, ihr_lo;  // inv_h_rho = inv_h_rhof + ihr_lo to double-float precision
};

// the factors of 1 / h_r = n / r_c, from the rounded quotient and its residue
inline void ne_split_inv_h(Tables& t, int n, double r_c)
{
    const double q = n / r_c;
    int ex;
    const double m = std::frexp(q, &ex);
    t.ih_hi = std::ldexp(std::nearbyint(std::ldexp(m, 29)), ex - 29);
    t.ih_k = ((q - t.ih_hi) + std::fma(-q, r_c, (double)n) / r_c) / t.ih_hi;
    t.ih_c = 0.5 + 0.5 * t.ih_k;
}

struct DevBatch {
    int n_rep, n_tot, n_tiles;
    int n_max;         // atoms of the largest replica
    int g;             // lanes per atom in the pair passes
    int sms;           // SMs of the device, and the most shared memory one of its blocks may have
    int smem_optin;
    const RepDev* rep;
    const int* tile_rep;
    double* x;
    double* v;
    const double* x0;
    float4* pos32;
    float4* posF;
    ned4* pos64;
    float4* pbuild;
    float4* csort;
    float4* f32;
    double* f64;
    double* rho;       // nullable: per-atom density output
    float* xi32;
    double* xi64;
    int* nbr;
    int* ncnt;
    int* sl;
    double* gs;        // FP64 path: [N][NE_SMAX]
    int* scnt;
    int* cellof;
    int* cslot;        // arrival order of each atom in its cell (list build)
    int* craw;         // atoms by cell, unsorted inside a cell (list build)
    int* cstart;
    int* ccount;       // atoms per cell; zero between list builds
    double* partA;     // [NPA][pair blocks], float2 (hi, lo) on the mixed path
    double* partB;     // [NPB][n_tiles], likewise
    double* partG;     // [NPA + NPB][n_grp] sums over groups of tiles
    int n_grp;
    unsigned* grp_done;
    double* tot;
    unsigned* tile_done;
    unsigned* nl_done;
    const double* lam; // lambda of the run's steps from lam_s0 on
    long long lam_s0;
    double* W;         // [n_rep][2]
    double* Wcum;      // nullable, [n_rep][2][t_s + 1]
    double* trace;     // nullable, [rows][8], single replica
    int trace_stride, trace_rows;
    int* flags;        // [n_rep] list rebuild requested (set by the step kernel)
    int* building;     // [n_rep] rebuild in progress (set by the binning, cleared by pass 1 or a run's set-up step)
    unsigned long long* rebuilds;  // count of replica list builds
    int* status;
    Tables tab;
    int npt_any;       // some replica has the barostat on (or the call wants the virial)
    int species_any;   // every replica has species tables (msd sampling per species)
};

// ------------------------------------------------------------------ lambda
// Sec. III.B: lambda = tau (function 1) or tau^5 (70 tau^4 - 315 tau^3 +
// 540 tau^2 - 420 tau + 126) (function 2); Sec. III.C: 1/(1 + tau(1/lf - 1)).
__host__ __device__ inline double ne_lambda_fl(int fn, double t)
{
    if (fn == 1) return t;
    double t2 = t * t;
    return t2 * t2 * t * (126.0 + t * (-420.0 + t * (540.0 + t * (-315.0 + t * 70.0))));
}

__host__ __device__ inline double ne_lambda_rs(double lf, double t)
{
    return 1.0 / (1.0 + t * (1.0 / lf - 1.0));
}

// Lambda in force at the start of global step s of the four-phase schedule.
__host__ __device__ inline double ne_sched_lambda(const Sched& S, long long s)
{
    if (S.kind == SCHED_FIXED) return s <= S.s0 ? S.lam_a : S.lam_b;
    const bool fl = S.path == 0;
    const double li = fl ? 0.0 : 1.0, lf = fl ? 1.0 : S.lambda_f;
    if (s <= S.t_eq) return li;
    long long s1 = s - S.t_eq;
    if (s1 <= S.t_s) {
        double tau = (double)s1 / (double)S.t_s;
        return fl ? ne_lambda_fl(S.fn, tau) : ne_lambda_rs(S.lambda_f, tau);
    }
    long long s2 = s1 - S.t_s;
    if (s2 <= S.t_eq) return lf;
    long long s3 = s2 - S.t_eq;
    if (s3 <= S.t_s) {
        double tau = (double)s3 / (double)S.t_s;
        return fl ? 1.0 - ne_lambda_fl(S.fn, tau) : ne_lambda_rs(S.lambda_f, 1.0 - tau);
    }
    return li;
}

// ------------------------------------------------------------------ Philox
// Philox4x32-10 (Salmon, Moraes, Dror & Shaw, SC'11): ten rounds, each two
// 32x32 -> 64-bit products mixed into the other words with the round key;
// the key advances by the Weyl increments between rounds.
__device__ __forceinline__ uint4 ne_philox(uint4 c, uint2 k)
{
    const uint32_t M0 = 0xD2511F53u, M1 = 0xCD9E8D57u;
    const uint32_t W0 = 0x9E3779B9u, W1 = 0xBB67AE85u;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        uint32_t hi0 = __umulhi(M0, c.x), lo0 = M0 * c.x;
        uint32_t hi1 = __umulhi(M1, c.z), lo1 = M1 * c.z;
        c = make_uint4(hi1 ^ c.y ^ k.x, lo1, hi0 ^ c.w ^ k.y, lo0);
        k.x += W0;
        k.y += W1;
    }
    return c;
}

__device__ __forceinline__ uint4 ne_philox_block(unsigned long long seed, unsigned replica,
                                                 unsigned stream, unsigned atom,
                                                 unsigned long long step)
{
    uint4 c = make_uint4(atom, (uint32_t)step, (uint32_t)(step >> 32), (replica << 4) | (stream & 15u));
    uint2 k = make_uint2((uint32_t)seed, (uint32_t)(seed >> 32));
    return ne_philox(c, k);
}

// Three standard normals from one Philox block by Box-Muller, uniforms
// (w + 1/2) 2^-32; the fourth normal is not used.
__device__ __forceinline__ void ne_normals64(uint4 w, double z[3])
{
    const double s = 2.3283064365386963e-10;  // 2^-32
    double u0 = ((double)w.x + 0.5) * s, u1 = ((double)w.y + 0.5) * s;
    double u2 = ((double)w.z + 0.5) * s, u3 = ((double)w.w + 0.5) * s;
    double r0 = sqrt(-2.0 * log(u0)), r1 = sqrt(-2.0 * log(u2));
    double s1, c1, s3, c3;
    sincospi(2.0 * u1, &s1, &c1);
    sincospi(2.0 * u3, &s3, &c3);
    z[0] = r0 * c1;
    z[1] = r0 * s1;
    z[2] = r1 * c3;
}

// FP32 variant: the top 24 bits of each word give u = (w>>8 + 1/2) 2^-24.
__device__ __forceinline__ void ne_normals32(uint4 w, float z[3])
{
    const float s = 5.9604644775390625e-8f;  // 2^-24
    float u0 = ((float)(w.x >> 8) + 0.5f) * s, u1 = ((float)(w.y >> 8) + 0.5f) * s;
    float u2 = ((float)(w.z >> 8) + 0.5f) * s, u3 = ((float)(w.w >> 8) + 0.5f) * s;
    float r0 = sqrtf(-2.0f * logf(u0)), r1 = sqrtf(-2.0f * logf(u2));
    float s1, c1, s3, c3;
    sincospif(2.0f * u1, &s1, &c1);
    sincospif(2.0f * u3, &s3, &c3);
    z[0] = r0 * c1;
    z[1] = r0 * s1;
    z[2] = r1 * c3;
}

// Component c of those normals alone, for one thread per component.
__device__ __forceinline__ double ne_normal64(uint4 w, int c)
{
    const double s = 2.3283064365386963e-10;  // 2^-32
    const double u0 = ((double)(c < 2 ? w.x : w.z) + 0.5) * s, u1 = ((double)(c < 2 ? w.y : w.w) + 0.5) * s;
    return sqrt(-2.0 * log(u0)) * (c == 1 ? sinpi(2.0 * u1) : cospi(2.0 * u1));
}

__device__ __forceinline__ float ne_normal32(uint4 w, int c)
{
    const float s = 5.9604644775390625e-8f;  // 2^-24
    const float u0 = ((float)((c < 2 ? w.x : w.z) >> 8) + 0.5f) * s, u1 = ((float)((c < 2 ? w.y : w.w) >> 8) + 0.5f) * s;
    float sn, cs;
    sincospif(2.0f * u1, &sn, &cs);
    return sqrtf(-2.0f * logf(u0)) * (c == 1 ? sn : cs);
}

// exp(x) - 1: the Taylor sum for the small arguments of a barostat step
// (|x| < 1/64: the eighth term is below 2^-57 of the first), else expm1
__device__ __forceinline__ double ne_baro_expm1(double x)
{
    if (fabs(x) >= 0.015625) return expm1(x);
    double t = fma(x, 1.0 / 5040.0, 1.0 / 720.0);
    t = fma(t, x, 1.0 / 120.0);
    t = fma(t, x, 1.0 / 24.0);
    t = fma(t, x, 1.0 / 6.0);
    t = fma(t, x, 0.5);
    return fma(t * x, x, x);
}

// ------------------------------------------------------------------ box
// x into [0, L) (w its FP32 copy; iL = 1 / L).  The image index is found in
// FP32, the shift, only for an atom outside the box, taken off in FP64 (one
// FMA's rounding).  The index of an atom N boxes away is off by up to N 2^-24,
// so what is left is wrapped again until it lies inside: once for an atom near
// the box, twice up to 2^24 boxes.  An atom beyond ~10^29 boxes stays outside.
__device__ __forceinline__ void ne_wrap(double& x, float& w, double L, float iL)
{
    w = (float)x;
#pragma unroll 1
    for (int k = 0; k < 4; ++k) {
        const float n = floorf(w * iL);
        if (n == 0.f) break;
        x = fma(-L, (double)n, x);
        w = (float)x;
    }
}

// ------------------------------------------------------------------ misc
// double-float (hi + lo, |lo| <= ulp(hi) / 2) sum of two such numbers from
// FP32 operations (TwoSum of the high parts, the low parts added to its error)
struct dff {
    float hi, lo;
};

__device__ __forceinline__ dff dff_add(dff a, dff b)
{
    const float s = a.hi + b.hi, bp = s - a.hi;
    float e = (a.hi - (s - bp)) + (b.hi - bp);
    e += a.lo + b.lo;
    const float h = s + e;
    return {h, e - (h - s)};
}

// sum over the warp of a double-float (fixed xor tree: every lane gets it)
__device__ __forceinline__ dff dff_warp_sum(dff v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1)
        v = dff_add(v, {__shfl_xor_sync(0xffffffffu, v.hi, o), __shfl_xor_sync(0xffffffffu, v.lo, o)});
    return v;
}

// Sum of nt consecutive partials, by one warp: lane l adds entries l, l + 32,
// ... in four interleaved chains, then a fixed xor-shuffle tree; every lane
// returns the total, and the order depends only on nt, never on scheduling.
// Called by all 32 lanes.  Partials are doubles on the FP64 path and
// double-float pairs, sixteen loads in flight, on the mixed one (serial FP64
// adds of a 65,536-atom replica's 2048 partials, 15 quantities in the one
// finishing block, cost 13 us).  A choice of fewer bits: such a sum of 16 to 2048
// partials is off by up to 3.4e-15 of it (an FP64 one by 1.5e-16), under terms that
// FP32 pairs leave at 1e-8 of it; the works are FP64.
__device__ __forceinline__ double ne_warp_part_sum(const double* part, int nt)
{
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    for (int t = threadIdx.x & 31; t < nt; t += 128)
#pragma unroll
        for (int c = 0; c < 4; ++c)
            if (t + 32 * c < nt) acc[c] += __ldcg(&part[t + 32 * c]);
    double s = (acc[0] + acc[1]) + (acc[2] + acc[3]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    return s;
}

__device__ __forceinline__ float2 ne_warp_part_sum_e(const float2* part, int nt)
{
    dff acc[4] = {};
    for (int t = threadIdx.x & 31; t < nt; t += 512) {
        float2 v[16];
#pragma unroll
        for (int c = 0; c < 16; ++c) v[c] = t + 32 * c < nt ? __ldcg(&part[t + 32 * c]) : make_float2(0.f, 0.f);
#pragma unroll
        for (int c = 0; c < 16; ++c)
            if (t + 32 * c < nt) acc[c & 3] = dff_add(acc[c & 3], {v[c].x, v[c].y});
    }
    const dff s = dff_warp_sum(dff_add(dff_add(acc[0], acc[1]), dff_add(acc[2], acc[3])));
    return make_float2(s.hi, s.lo);
}

__device__ __forceinline__ double ne_warp_part_sum_e(const double* part, int nt) { return ne_warp_part_sum(part, nt); }

__device__ __forceinline__ double ne_warp_part_sum(const float2* part, int nt)
{
    const float2 s = ne_warp_part_sum_e(part, nt);
    return (double)s.x + (double)s.y;
}

// nt partials from entry `at` of a partials array of either kind
__device__ __forceinline__ double ne_warp_part_sum(const DevBatch& B, const double* part, size_t at, int nt)
{
    return B.pos64 ? ne_warp_part_sum(part + at, nt) : ne_warp_part_sum((const float2*)part + at, nt);
}

// One more on a ticket, after this thread's earlier writes (and, behind a
// barrier, its block's); returns the count before.  A release only:
// __threadfence also drops the SM's L1, which the blocks next to a finishing
// one pay for.
__device__ __forceinline__ unsigned ne_ticket(unsigned* p)
{
    unsigned old;
    asm volatile("atom.release.gpu.global.add.u32 %0, [%1], 1;" : "=r"(old) : "l"(p) : "memory");
    return old;
}

// The kernels of a step follow one another in a stream, each reading what the
// one before wrote.  They are launched with ne_launch, which lets a kernel's
// blocks take their places on the SMs while the one before drains; every one
// of its threads calls ne_chain before it reads what an earlier kernel of the
// chain writes, and before it returns (a kernel that ended without having
// waited would let the next one pass its wait too early).  Before it a thread
// reads only what is fixed for the whole call: the tiles' replicas, the replica
// table but for a barostatted box.  The chain's first kernel, k_nl_cells, reads
// nothing before its wait: the kernel before it (k_setup, which writes both
// tables) is launched plainly and lets it in when its blocks end, but its
// writes are sure to be seen only behind the wait.  A later kernel begins after
// the wait of the one before it, and so after every write of that set-up.  The next
// kernel is let in after the wait: let in before it, the step kernel's normals
// ran beside pass 1 and took its FP64 slots (15.8 ms against 16.6 to 19.8,
// with the SMs that the blocks fell on, for the 600 steps of 128 atoms).
// What bounds a step of a small replica are the latencies of five kernels and
// the gaps between them: 128 atoms in FP64, replayed from a graph, 33.1 -> 25.8
// us a step; 2000 atoms launched one by one 35 -> 22 us; 65,536 atoms with the
// parameter gradient 155 -> 149 us.
__device__ __forceinline__ void ne_chain()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <typename... P, typename... A>
inline cudaError_t ne_launch(void (*k)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, const A&... a)
{
    cudaLaunchAttribute at = {};
    at.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t c = {};
    c.gridDim = grid;
    c.blockDim = block;
    c.dynamicSmemBytes = smem;
    c.stream = st;
    c.attrs = &at;
    c.numAttrs = 1;
    return cudaLaunchKernelEx(&c, k, P(a)...);
}

__device__ __forceinline__ void ne_set_status(int* status, int bits)
{
    atomicOr(status, bits);
}

// Launch helpers (defined in the kernel translation units).
namespace ne {
void launch_tables(const double* theta, int nk, double r_c, double rho_max, float4* pf32,
                   ned4* pf64, float4* F32, ned4* F64, cudaStream_t st);
// list build of the flagged (or, forced, all) replicas around the sites (the
// step kernel then writes the positions for the pair passes) or the positions
// (written here)
void launch_nl_build(const DevBatch& B, int force, int from_sites, cudaStream_t st);
int lanes_per_atom(int n_tot);  // the pair passes' lanes per atom for a batch of n_tot atoms
void launch_pass1(const DevBatch& B, bool mixed, cudaStream_t st);
void launch_pass2(const DevBatch& B, bool mixed, cudaStream_t st);
// (0, 0): no kick and no step, the copies, sums and normals of the first step
void launch_step(const DevBatch& B, const Sched& S, bool mixed, const long long* step_base,
                 int j, int do_close, int do_open, cudaStream_t st);
constexpr int SETUP_REPS = 6;    // replicas a set-up launch takes (their table is its argument: 4 KB)
// Replicas up to which the set-up goes by launches, above by copies and clears.  A
// run of no steps in us by the one and the other: 1 replica 30, 35; 6 38, 45; 12 51,
// 53; 24 72, 70; 36 94, 86; 72 164, 134
constexpr int SETUP_MAX = 24;
void launch_setup(const RepDev* reps, int n_rep, RepDev* rep, int* tile_rep, unsigned* tile_done, int* flags,
                  int* status, double* tot, cudaStream_t st);
cudaError_t launch_status_out(const int* status, int* host, cudaStream_t st);  // host: pinned
void launch_set_step(long long* step_base, long long s, cudaStream_t st);
void launch_advance(long long* step_base, long long by, cudaStream_t st);
void launch_noise(unsigned long long seed, unsigned replica, int stream, long long step, int n, int mixed,
                  double* z, cudaStream_t st);
void launch_init_velocities(const DevBatch& B, int fix_cm, cudaStream_t st);
void launch_spring(const double* x, const double* x0, int n, double k, double* f, double* e,
                   double* scratch, cudaStream_t st);
void launch_export(const DevBatch& B, bool mixed, double* f_out, double* e_out, double scale, cudaStream_t st);
void launch_msd_sample(const DevBatch& B, double* acc, cudaStream_t st);
// gE, or with gw != nullptr the per-step weight gw[*ctr + j - s_off] read on
// the device (runs replayed from graphs); set_attr: set the kernel's shared-
// memory attribute (not inside a stream capture)
size_t backward_bins_bytes(int nk);   // the mixed backward's global bins, zero between launches
bool backward_fits(int nk);           // a block's low words fit its shared memory
void launch_backward(const DevBatch& B, bool mixed, double gE, double* gtheta,
                     unsigned long long* bins, bool accumulate, cudaStream_t st,
                     const double* gw = nullptr, const long long* ctr = nullptr, int j = 0,
                     long long s_off = 0, bool set_attr = true);
cudaError_t prepare_backward(const DevBatch& B);  // the mixed backward kernel's shared-memory attribute
void launch_virial(const DevBatch& B, double* out, cudaStream_t st);
}  // namespace ne
