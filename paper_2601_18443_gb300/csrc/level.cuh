// level.cuh -- sm_103a kernels of one LBM-RANS level step (included by one source file per
// storage type, and by kernels.cu for the code it shares).
//
// Populations are stored shifted, g_q = f_q - w_q, as structure of arrays over the level's 32 x 8
// tiles; a warp works on the cells of 16 x 2 blocks of a tile.  The collision is the
// central-moment operator of eqs 5-7 evaluated in closed form on the shifted raw moments
// (rest-state moments subtracted analytically), so that FP32 keeps the small departures from rest
// exact to ~1e-7 relative.  No step is a dense contraction; large levels are bound by memory
// bandwidth, small ones by the latency of one warp.
//
// One launch of k_level advances every active cell of a level by one level step:
// wall function of its boundary node (finest level, Sec 2.3 steps 1-5), SA-neg
// update of chi (Sec 2.2), pull streaming with coalescence from the finer level and
// Yu's slip bounce-back on cut links (eq 27), central-moment collision relaxing with
// nu + nu_t, explosion into the finer level's ghosts, and -- on the second sub-step
// of a level -- the restriction of the new fields into the covered parents.  Fields
// of time t are read from buffer [p] and those of t + 1 written to [p ^ 1], so that
// no cell reads a value another block of the same launch writes.
#pragma once

#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <math.h>

#include <type_traits>

#include "device.cuh"

namespace lbmdev {

// ------------------------------------------------------------------ lattice (eq 2)
__host__ __device__ constexpr int cxq(int q) { return q == 1 || q == 5 || q == 7 ? 1 : (q == 2 || q == 6 || q == 8 ? -1 : 0); }
__host__ __device__ constexpr int cyq(int q) { return q == 3 || q == 5 || q == 8 ? 1 : (q == 4 || q == 6 || q == 7 ? -1 : 0); }
__host__ __device__ constexpr int oppq(int q) { return q == 0 ? 0 : (q & 1 ? q + 1 : q - 1); }
__host__ __device__ constexpr float wq(int q) { return q == 0 ? 4.f / 9.f : (q < 5 ? 1.f / 9.f : 1.f / 36.f); }
// direction with the same c_x and the opposite c_y (specular reflection on a horizontal plane)
__host__ __device__ constexpr int mirror_y(int q)
{
    return q == 3 ? 4 : q == 4 ? 3 : q == 5 ? 7 : q == 7 ? 5 : q == 6 ? 8 : q == 8 ? 6 : q;
}
// D2Q9 index of the offset (sx, sy) stored at position (sy + 1) * 3 + (sx + 1)
__host__ __device__ constexpr int dir_of3(int m)
{
    return m == 4 ? 0 : m == 5 ? 1 : m == 3 ? 2 : m == 7 ? 3 : m == 1 ? 4 : m == 8 ? 5 : m == 0 ? 6 : m == 2 ? 7 : 8;
}

// The 3 x 3 block of tiles around the block's tile, staged in shared memory.
__device__ __forceinline__ void load_nb3(const LevelView &P, int t, int *nb3)
{
    if (threadIdx.x < 9) nb3[threadIdx.x] = P.nbr[t * 9 + dir_of3(threadIdx.x)];
}

// Thread -> cell map of a tile: warp w covers the 16 x 2 cells x in [16 (w & 1), +16), y in
// {2 (w >> 1), +1}, so that every 2 x 2 group of children lies inside one warp (the restriction
// is a warp shuffle) and a warp reads two 64-byte row segments per plane.
__device__ __forceinline__ void cell_of_thread(int c, int &lx, int &ly)
{
    const int w = c >> 5, lane = c & 31;
    lx = (w & 1) * 16 + (lane & 15);
    ly = (w >> 1) * 2 + (lane >> 4);
}

// The slots of the eight D2Q9 neighbours at offsets +c_q (q = 1..8) and the own slot
// (q = 0); a neighbour in an absent tile maps to the own slot and clears bit q of the
// returned presence mask.  The SA stencil reads offset +c_q, the pull of direction q
// reads offset -c_q = +c_opp(q).
__device__ __forceinline__ unsigned neighbours(const int *nb3, int lx, int ly, int slot, int nbs[9])
{
    const int xm = lx - 1, xp = lx + 1, ym = ly - 1, yp = ly + 1;
    const int cm = xm < 0 ? 0 : 1, cp = xp >= LBM_TX ? 2 : 1;              // tile column of x -/+ 1
    const int rm = ym < 0 ? 0 : 3, rp = yp >= LBM_TY ? 6 : 3;              // tile row (x 3) of y -/+ 1
    const int colm = xm & (LBM_TX - 1), colp = xp & (LBM_TX - 1);
    const int rowm = (ym & (LBM_TY - 1)) * LBM_TX, rowp = (yp & (LBM_TY - 1)) * LBM_TX, row0 = ly * LBM_TX;
    const int tl[9] = {0, nb3[3 + cp], nb3[3 + cm], nb3[rp + 1], nb3[rm + 1], nb3[rp + cp], nb3[rm + cm],
                       nb3[rm + cp], nb3[rp + cm]};
    const int off[9] = {0, row0 + colp, row0 + colm, rowp + lx, rowm + lx, rowp + colp, rowm + colm, rowm + colp,
                        rowp + colm};
    unsigned present = 1u;
    nbs[0] = slot;
#pragma unroll
    for (int q = 1; q < 9; q++) {
        const bool ok = tl[q] >= 0;
        nbs[q] = ok ? tl[q] * LBM_TILE + off[q] : slot;
        present |= ok ? (1u << q) : 0u;
    }
    return present;
}

// level 0 covers its whole box with tiles in row-major order
__device__ __forceinline__ int slot0(const StepConsts &k, int i, int j)
{
    return ((j >> 3) * k.ntx0 + (i >> 5)) * LBM_TILE + (j & 7) * LBM_TX + (i & 31);
}

// the tile of level l+1 holding the four children of (lx, ly) and their first slot
__device__ __forceinline__ int child_base(const LevelView &P, int t, int lx, int ly)
{
    const int ct = P.child[t * 4 + ((2 * ly) >> 3) * 2 + ((2 * lx) >> 5)];
    return ct < 0 ? -1 : ct * LBM_TILE + ((2 * ly) & 7) * LBM_TX + ((2 * lx) & 31);
}

// ------------------------------------------------------------------ population storage
// Populations are stored shifted (f - w) in FP32, FP16 or BF16; every load converts to
// FP32 and every store rounds to nearest, so the arithmetic is FP32 in all three forms.
template <typename T> struct PopIO;
template <> struct PopIO<float> {
    static __device__ __forceinline__ float ld(const float *p) { return *p; }
    static __device__ __forceinline__ void st(float *p, float v) { *p = v; }
};
template <> struct PopIO<__half> {
    static __device__ __forceinline__ float ld(const __half *p) { return __half2float(*p); }
    static __device__ __forceinline__ void st(__half *p, float v) { *p = __float2half_rn(v); }
};
template <> struct PopIO<__nv_bfloat16> {
    static __device__ __forceinline__ float ld(const __nv_bfloat16 *p) { return __bfloat162float(*p); }
    static __device__ __forceinline__ void st(__nv_bfloat16 *p, float v) { *p = __float2bfloat16_rn(v); }
};

// two consecutive stored populations as one access
__device__ __forceinline__ float2 pop_ld2(const float *p) { return *reinterpret_cast<const float2 *>(p); }
__device__ __forceinline__ float2 pop_ld2(const __half *p) { return __half22float2(*reinterpret_cast<const __half2 *>(p)); }
__device__ __forceinline__ float2 pop_ld2(const __nv_bfloat16 *p)
{
    return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(p));
}
__device__ __forceinline__ void pop_st2(float *p, float a, float b) { *reinterpret_cast<float2 *>(p) = make_float2(a, b); }
__device__ __forceinline__ void pop_st2(__half *p, float a, float b) { *reinterpret_cast<__half2 *>(p) = __floats2half2_rn(a, b); }
__device__ __forceinline__ void pop_st2(__nv_bfloat16 *p, float a, float b)
{
    *reinterpret_cast<__nv_bfloat162 *>(p) = __floats2bfloat162_rn(a, b);
}

// asynchronous copy of N bytes (4 or 8, aligned to N) from global to the thread's own shared
// memory; own copies can be read after async_wait
template <int N> __device__ __forceinline__ void async_copy(void *dst, const void *src)
{
    const unsigned d = (unsigned)__cvta_generic_to_shared(dst);
    asm volatile("cp.async.ca.shared.global [%0], [%1], %2;" ::"r"(d), "l"(src), "n"(N) : "memory");
}
__device__ __forceinline__ void async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// ------------------------------------------------------------------ programmatic dependent launch
// The level-step kernels are launched with programmatic stream serialization: the next
// kernel's blocks may be scheduled while this one drains.  Each kernel reads only
// static tables before griddep_wait(), which returns once the preceding kernel has
// completed and its writes are visible; griddep_launch() lets the next kernel start
// being scheduled as soon as every block of this one has begun.  What a preceding kernel may
// have written is read with ordinary loads: __ldg tells the compiler that the value never
// changes, and it then moves the load up across the wait.
__device__ __forceinline__ void griddep_wait()
{
    asm volatile("griddepcontrol.wait;" ::: "memory");
}

__device__ __forceinline__ void griddep_launch()
{
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

// ------------------------------------------------------------------ launch timeline
// With a timeline buffer (lbm_set_timeline), thread 0 of each block records the global
// timer (ns) at the block's entry, once its wait for the preceding kernel has returned, and
// once all its threads are done, at tl[3 (base + block) + 0, 1, 2].  Without one (tl null,
// a kernel parameter, so every branch here is uniform) nothing is read or written.
__device__ __forceinline__ void tl_mark(unsigned long long *tl, int base, int m)
{
    if (tl != nullptr && threadIdx.x == 0) {
        unsigned long long t;
        asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
        tl[3ull * (unsigned)(base + (int)blockIdx.x) + (unsigned)m] = t;
    }
}

__device__ __forceinline__ void tl_end(unsigned long long *tl, int base)
{
    if (tl == nullptr) return;
    __syncthreads();
    tl_mark(tl, base, 2);
}

// ------------------------------------------------------------------ bounds-checked builds
// With LBM_BOUNDS_CHECK every index the level step follows from a table (the work lists,
// tile neighbours, children and parents, the aux word, the wall stencils) is checked
// against its buffer: one outside it sets LBM_STATUS_BOUNDS in the status word (when the
// caller has one) and is replaced by 0, so that the access stays inside the buffer and no
// lane leaves its warp early; the host then fails the next synchronising call.  The default
// build compiles none of it.
__device__ __forceinline__ int checked_index(int i, int n, int *status)
{
#ifdef LBM_BOUNDS_CHECK
    if (i < 0 || i >= n) {
        if (status) atomicOr(status, LBM_STATUS_BOUNDS);
        return 0;
    }
#else
    (void)n;
    (void)status;
#endif
    return i;
}

// ------------------------------------------------------------------ SA-neg constants (Sec 2.2)
#define SA_CB1 0.1355f
#define SA_CB2 0.622f
#define SA_SIGMA (2.0f / 3.0f)
#define SA_KAPPA 0.41f
#define SA_CW1 3.2390678f             /* cb1 / kappa^2 + (1 + cb2) / sigma */
#define SA_CW2 0.3f
#define SA_CW3_6 64.0f                /* cw3^6, cw3 = 2 */
#define SA_CV1_3 357.911f             /* cv1^3, cv1 = 7.1 */
#define SA_RLIM 10.0f
#define SA_CV2 0.7f
#define SA_CV3 0.9f                   /* reading: value of the SA-neg source the paper follows */
#define SA_CT3 1.2f
#define SA_CN1 16.0f

// ------------------------------------------------------------------ collision (eqs 5-10)
// Input: post-stream shifted populations g (f - w).  Output: post-collision shifted
// populations.  drho, jx, jy: the conserved moments of eq 3 summed from g; ux, uy the
// velocity j / rho.  The conserved raw moments are taken from the sums themselves, so
// mass and momentum are conserved to the rounding of those sums whatever the rounding
// of u.  delta = 2 - omega_nu (omega_b = 1: the trace relaxes fully, Sec 2.1).
__device__ __forceinline__ void collide_cm(const float g[9], float drho, float jx, float jy, float ux, float uy,
                                           float delta, float o[9])
{
    const float rho = 1.0f + drho;
    const float m20 = g[1] + g[2] + g[5] + g[6] + g[7] + g[8];   // sum cx^2 g  (= m20 - 1/3)
    const float m02 = g[3] + g[4] + g[5] + g[6] + g[7] + g[8];   // sum cy^2 g
    const float m11 = g[5] + g[6] - g[7] - g[8];
    const float uxx = ux * ux, uyy = uy * uy, uxy = ux * uy;
    const float D = (m20 - m02) - rho * (uxx - uyy);              // k20 - k02
    const float K = m11 - rho * uxy;                              // k11
    const float Ds = delta * D - D;                               // (1 - omega) (k20 - k02)
    const float Ks = delta * K - K;                               // (1 - omega) k11
    const float k20 = rho * (1.0f / 3.0f) + 0.5f * Ds;            // post-collision central moments
    const float k02 = rho * (1.0f / 3.0f) - 0.5f * Ds;
    // raw post-collision moments minus their rest-state values (binomial shift back)
    const float M00 = drho;
    const float M10 = jx, M01 = jy;
    const float M20 = drho * (1.0f / 3.0f) + 0.5f * Ds + rho * uxx;
    const float M02 = drho * (1.0f / 3.0f) - 0.5f * Ds + rho * uyy;
    const float M11 = Ks + rho * uxy;
    const float M21 = uy * k20 + 2.0f * ux * Ks + rho * uxx * uy;
    const float M12 = ux * k02 + 2.0f * uy * Ks + rho * ux * uyy;
    const float M22 = drho * (1.0f / 9.0f) + uyy * k20 + uxx * k02 + 4.0f * uxy * Ks + rho * uxx * uyy;
    // populations from the nine raw moments of D2Q9
    o[0] = M00 - M20 - M02 + M22;
    o[1] = 0.5f * (M10 + M20 - M12 - M22);
    o[2] = 0.5f * (-M10 + M20 + M12 - M22);
    o[3] = 0.5f * (M01 + M02 - M21 - M22);
    o[4] = 0.5f * (-M01 + M02 + M21 - M22);
    o[5] = 0.25f * (M11 + M21 + M12 + M22);
    o[6] = 0.25f * (M11 - M21 - M12 + M22);
    o[7] = 0.25f * (-M11 - M21 + M12 + M22);
    o[8] = 0.25f * (-M11 + M21 - M12 + M22);
}

// 2 - omega for the effective viscosity nu + nu_t (eq 9 with the RANS substitution);
// the divisions use the fast reciprocal path (about 2 ulp)
__device__ __forceinline__ float delta_of(float nu, float chi, int turbulence)
{
    float nue = nu;
    if (turbulence) {
        const float c3 = chi * chi * chi;
        nue += fmaxf(chi, 0.0f) * nu * __fdividef(c3, c3 + SA_CV1_3);
    }
    return __fdividef(12.0f * nue, 1.0f + 6.0f * nue);
}

// ------------------------------------------------------------------ SA-neg (Sec 2.2)
struct Stencil {
    float chi[9], ux[9], uy[9];
};

// level-0 box edge: neighbours across the top/bottom symmetry planes are mirror images
__device__ __forceinline__ void gather0(const float *chi, const float *ux, const float *uy, const StepConsts &k, int i,
                                        int j, Stencil &S)
{
#pragma unroll
    for (int q = 0; q < 9; q++) {
        int ii = i + cxq(q), jj = j + cyq(q);
        float sg = 1.0f;
        if (jj < 0) { jj = 0; sg = -1.0f; }
        if (jj >= k.ny0) { jj = k.ny0 - 1; sg = -1.0f; }
        if (ii < 0) ii = 0;
        if (ii >= k.nx0) ii = k.nx0 - 1;
        const int s = slot0(k, ii, jj);
        S.chi[q] = chi[s]; S.ux[q] = ux[s]; S.uy[q] = sg * uy[s];
    }
}

// LSQ gradient over the full D2Q9 neighbourhood: the normal matrix is 6 I, so the
// gradient is sum_k c_k (phi_k - phi_0) / 6 = sum_k c_k phi_k / 6 (sum_k c_k = 0)
__device__ __forceinline__ void lsq_grad(const float *v, float &gx, float &gy)
{
    gx = ((v[1] - v[2]) + (v[5] - v[6]) + (v[7] - v[8])) * (1.0f / 6.0f);
    gy = ((v[3] - v[4]) + (v[5] - v[6]) + (v[8] - v[7])) * (1.0f / 6.0f);
}

__device__ __forceinline__ float sa_diff_coef(float chi)
{   // (nu + nu_t~ f_n) / nu
    const float c3 = chi * chi * chi;
    const float fn = chi < 0.0f ? __fdividef(SA_CN1 + c3, SA_CN1 - c3) : 1.0f;
    return 1.0f + chi * fn;
}

// Euler step of eqs 12 / 16 written for chi = nu_t~ / nu (explicit, with the diagonal of the
// diffusion at the new time level), with Lax-Wendroff (conv = 0, Sec 2.2) or first-order
// upwind (conv = 1, Sec 3.3) convection;
// vort the magnitude of the vorticity, POS: chi is known not to be negative at the centre and its
// four face neighbours, id2 = 1 / d^2 (wall distance d in level lattice units)
template <bool POS>
__device__ __forceinline__ float sa_point(const float x[9], float u, float v, float vort, float id2, float nu, int conv)
{
    // x: 0 C, 1 E, 2 W, 3 N, 4 S, 5 NE, 6 SW, 7 SE, 8 NW
    const float gx = 0.5f * (x[1] - x[2]), gy = 0.5f * (x[3] - x[4]);
    const float gxx = x[1] - 2.0f * x[0] + x[2], gyy = x[3] - 2.0f * x[0] + x[4];
    const float gxy = 0.25f * (x[5] - x[8] - x[7] + x[6]);
    const float cv = conv == 1
                         ? -(u * (u > 0.0f ? x[0] - x[2] : x[1] - x[0]) + v * (v > 0.0f ? x[0] - x[4] : x[3] - x[0]))
                         : -(u * gx + v * gy) + 0.5f * (u * u * gxx + 2.0f * u * v * gxy + v * v * gyy);
    float Dc, De, Dw, Dn, Ds;
    if (POS || fminf(fminf(x[0], x[1]), fminf(fminf(x[2], x[3]), x[4])) >= 0.0f) {
        // nu_t~ >= 0 on the whole stencil: f_n = 1
        Dc = 1.0f + x[0];
        De = 0.5f * (Dc + 1.0f + x[1]); Dw = 0.5f * (Dc + 1.0f + x[2]);
        Dn = 0.5f * (Dc + 1.0f + x[3]); Ds = 0.5f * (Dc + 1.0f + x[4]);
    } else {
        Dc = sa_diff_coef(x[0]);
        De = 0.5f * (Dc + sa_diff_coef(x[1])); Dw = 0.5f * (Dc + sa_diff_coef(x[2]));
        Dn = 0.5f * (Dc + sa_diff_coef(x[3])); Ds = 0.5f * (Dc + sa_diff_coef(x[4]));
    }
    const float div = De * (x[1] - x[0]) - Dw * (x[0] - x[2]) + Dn * (x[3] - x[0]) - Ds * (x[0] - x[4]);
    const float diff = nu * (div + SA_CB2 * (gx * gx + gy * gy)) * (1.0f / SA_SIGMA);
    const float chi = x[0];
    const float ikd2 = id2 * (1.0f / (SA_KAPPA * SA_KAPPA));      // 1 / (kappa d)^2
    float src;
    if (POS || chi >= 0.0f) {
        const float c3 = chi * chi * chi;
        const float fv1 = __fdividef(c3, c3 + SA_CV1_3);
        const float fv2 = 1.0f - __fdividef(chi, 1.0f + chi * fv1);
        const float sbar = nu * chi * fv2 * ikd2;
        float st;
        if (sbar >= -SA_CV2 * vort) st = vort + sbar;
        else st = vort + __fdividef(vort * (SA_CV2 * SA_CV2 * vort + SA_CV3 * sbar), (SA_CV3 - 2.0f * SA_CV2) * vort - sbar);
        float r = SA_RLIM;
        if (st > 0.0f) r = fminf(__fdividef(nu * chi * ikd2, st), SA_RLIM);
        const float r2 = r * r, r6 = r2 * r2 * r2;
        const float gg = r + SA_CW2 * (r6 - r);
        const float g2 = gg * gg, g6 = g2 * g2 * g2;
        const float fw = gg * __powf(__fdividef(1.0f + SA_CW3_6, g6 + SA_CW3_6), 1.0f / 6.0f);
        src = SA_CB1 * st * chi - SA_CW1 * fw * nu * chi * chi * id2;
    } else {
        src = SA_CB1 * (1.0f - SA_CT3) * vort * chi + SA_CW1 * nu * chi * chi * id2;
    }
    // the diffusion's diagonal at the new time level (point-implicit): the explicit increment
    // divided by 1 + sum_f D_f / sigma; unconditionally stable diffusion, same steady states
    const float a = nu * (De + Dw + Dn + Ds) * (1.0f / SA_SIGMA);
    return chi + __fdividef(cv + src + diff, 1.0f + a);
}

__device__ __forceinline__ float sa_update(const Stencil &S, float id2, float nu, int conv)
{
    float dudx, dudy, dvdx, dvdy;
    lsq_grad(S.ux, dudx, dudy);
    lsq_grad(S.uy, dvdx, dvdy);
    return sa_point<false>(S.chi, S.ux[0], S.uy[0], fabsf(dvdx - dudy), id2, nu, conv);
}

// ------------------------------------------------------------------ wall function (Sec 2.3 steps 1-5)
#define WF_B 5.033908790505579f
#define WF_A1 8.148221580024245f
#define WF_A2 (-6.9287093849022945f)
#define WF_B1 7.4600876082527945f
#define WF_B2 7.468145790401841f
#define WF_C1 2.5496773539754747f
#define WF_C2 1.3301651588535228f
#define WF_C3 3.599459109332379f
#define WF_C4 3.639753186868684494f

__device__ __forceinline__ float wf_uplus(float y)
{   // eq 22 on the continuous arctangent branch: with b > 0, atan2(b, x) = pi/2 - atan(x / b)
    const float z1 = (y + WF_A1) * (1.0f / WF_B1), z2 = (y + WF_A2) * (1.0f / WF_B2);
    const float t1 = (y + WF_A1) * (y + WF_A1) + WF_B1 * WF_B1;
    const float t2 = (y + WF_A2) * (y + WF_A2) + WF_B2 * WF_B2;
    return (WF_B - (WF_C3 + WF_C4) * 1.5707963267948966f) + WF_C1 * __logf(t1) - WF_C2 * __logf(t2) +
           WF_C3 * atanf(z1) + WF_C4 * atanf(z2);
}

__device__ __forceinline__ float wf_dudy(float y)
{   // eq 21
    float k3 = SA_KAPPA * y;
    k3 = k3 * k3 * k3;
    return __fdividef(SA_CV1_3 + k3, SA_CV1_3 + k3 * (1.0f + SA_KAPPA * y));
}

// Friction velocity from u_t at distance y (step 3): the root of g(u) = u u+(u y / nu) - u_t,
// g' = u+ + y+ du+/dy+ > 0, started from the previous sub-step's value when there is one, else
// from the viscous-sublayer value.  y_nu = y / nu.  While g is far from zero (more than 5 % of
// u_t) the step is Newton's in the logarithms, u (u_t / (u u+))^(u+ / g'): u u+ is a power of u
// whose exponent g' / u+ only varies from 2 (viscous sublayer) to about 1.1 (log layer), so a
// start off by a factor of ten takes two or three such steps where Newton's own halves its
// distance per step.  Near the root it is Newton's own step, and the iteration stops after one
// shorter than 3e-4 u: its error after a step of relative size e is about (g'' u / 2 g') e^2, at
// most e^2 / 2 (the viscous sublayer; about 0.05 e^2 in the log layer), so the result is within
// 4.5e-8 relative of the root, below FP32 resolution.  It also stops where g is within the
// rounding of u+ (terms of up to 20 in FP32: 4e-6), which below y+ of about 0.01 is more than 3e-4
// of u+: without that rule the few boundary nodes near a stagnation point ran through the limit
// of evaluations in every step, and the whole launch waited for them.  Over u_t from 1e-9 to 0.5
// and y / nu from 10 to 3e6 it takes one evaluation from the previous step's value, two after
// that has moved by 1e-3, at most six from anywhere (limit 24).
__device__ __forceinline__ float wf_utau(float ut, float y_nu, float guess)
{
    if (!(ut > 0.0f)) return 0.0f;
    float u = guess > 0.0f ? guess : sqrtf(ut / y_nu);
    for (int it = 0; it < 24; it++) {
        const float yp = u * y_nu;
        const float up = wf_uplus(yp);
        const float gv = u * up - ut;
        const float gp = up + yp * wf_dudy(yp);
        if (fabsf(gv) > 0.05f * ut) {
            u *= __powf(__fdividef(ut, u * up), __fdividef(up, gp));
            continue;
        }
        const float un = u - __fdividef(gv, gp);
        const bool done = fabsf(un - u) <= 3e-4f * un || fabsf(gv) <= 4e-6f * u;
        u = un;
        if (done) break;
    }
    return u;
}

// Step 1 of Sec 2.3 over one row of a record's 4 x 4 stencil (unused entries carry zero weight):
// rho_R - 1 and u_R as weighted sums of the fields at time level p.
__device__ __forceinline__ void wall_gather(const LevelView &P, int p, int4 sv, float4 wr, float4 wu, float &drR, float &uR,
                                            float &vR, int *status)
{
    const float *dr = P.drho[p], *ux = P.ux[p], *uy = P.uy[p];
    const int sa[4] = {sv.x, sv.y, sv.z, sv.w};
    const float ra[4] = {wr.x, wr.y, wr.z, wr.w}, ua[4] = {wu.x, wu.y, wu.z, wu.w};
#pragma unroll
    for (int m = 0; m < 4; m++) {
        const int s = checked_index(sa[m], P.ns, status);
        drR += ra[m] * dr[s]; uR += ua[m] * ux[s]; vR += ua[m] * uy[s];
    }
}

struct WallState {
    float uWx, uWy, utau, chiB, tx, ty, ut;
};

// Steps 2-5 of Sec 2.3 for one boundary node from the velocity at R (tangential part, u_tau from
// eq 22 by Newton from `start`, u_V, slip velocity of eq 28 along t) and the SA Dirichlet value
// (Sec 2.2).
__device__ __forceinline__ WallState wall_point(const LevelView &P, const RecView &R, const StepConsts &k, int r, float nx,
                                                float ny, float dwb, float start, float uR, float vR)
{
    const float inu = 1.0f / P.nu;
    const float un = uR * nx + vR * ny;
    const float utx = uR - un * nx, uty = vR - un * ny;
    WallState w;
    w.ut = sqrtf(utx * utx + uty * uty);
    w.tx = -ny; w.ty = nx;
    if (w.ut > 0.0f) { const float iut = 1.0f / w.ut; w.tx = utx * iut; w.ty = uty * iut; }
    w.utau = 0.f; w.uWx = 0.f; w.uWy = 0.f; w.chiB = 0.f;
    if (k.wall_model < 2) {
        w.utau = wf_utau(w.ut, k.d_wr * inu, start);                                // step 3
        float uW;
        if (k.wall_model == 0) {
            const float ypv = w.utau * k.d_wv * inu;
            const float uV = w.utau * wf_uplus(ypv);                                // step 4
            uW = uV - __fdividef(w.utau * w.utau * k.d_wv * inu, 1.0f + SA_KAPPA * ypv);   // eq 28
        } else {
            // Nishimura's slip adapted to RANS (Sec 3.1.5, eq 31): the slip extrapolated linearly
            // from R with the SA log-layer eddy viscosity (nu_t)_R = nu kappa y+_R (eq 20)
            const float ypr = w.utau * k.d_wr * inu;
            uW = w.ut - __fdividef(w.utau * w.utau * k.d_wr * inu, 1.0f + SA_KAPPA * ypr);
        }
        w.uWx = uW * w.tx; w.uWy = uW * w.ty;                                       // step 5
        w.chiB = SA_KAPPA * w.utau * dwb * inu;
    } else if (k.wall_model == 2) {
        w.uWx = R.slip[2 * R.loop[r]]; w.uWy = R.slip[2 * R.loop[r] + 1];
    }
    return w;
}

// ------------------------------------------------------------------ the fused level step
// Population layout (one lattice per level, updated in place; the "AA pattern").  With
// d the storage direction of a slot and q the population it holds:
//   before an even step (p = 0) slot (x, q) holds the population f_q arriving at x,
//   before an odd step  (p = 1) slot (x, opp q) holds the post-collision f*_q of x.
// An even step reads its cell's own nine slots and writes f*_q to (x, opp q).  An odd
// step reads f*_q of the upstream cell from (x - c_q, opp q) and writes its own f*_q to
// (x + c_q, q), the slot the downstream cell reads in the next even step.  In either
// step each slot is read and then written by one thread only (its own cell in an even
// step, the cell x - c_q of slot (x, q) in an odd step), so one lattice suffices.
// Levels l >= 1 take their two sub-steps of a parent step as an even and an odd step;
// level 0 alternates from coarse step to coarse step.
//
// Values that a step needs but that another thread's slot holds are kept in small side
// buffers written by the cell that owns them:
//   - a boundary node's last post-collision populations (R.fpost), for eq 27;
//   - the outlet columns' post-collision populations entering from x = N (k.obuf);
//   - a band cell's last post-collision populations (ebuf: the explosion), which its ghost
//     children keep where their upstream cell is not fluid;
//   - the populations each ghost child pulled in the fine level's odd sub-step (gbuf), which
//     the band cell averages (the coalescence).
// 16-bit storage keeps populations relative to the free-stream equilibrium, so that in
// most of the domain the stored values are small and their relative rounding is small in
// absolute terms; FP32 storage keeps g = f - w itself.  The shift belongs to the population
// (q), not to the slot direction (d).
// Slot (d, s) is element d * ns + s: a 32-bit index, since the host keeps 9 ns below 2^31.
template <typename T> struct Lat {
    T *f;
    int ns;
    const float *sh;
    __device__ __forceinline__ float ld(int d, int s, int q) const
    {
        if constexpr (std::is_same<T, float>::value) return PopIO<T>::ld(f + (d * ns + s));
        else return PopIO<T>::ld(f + (d * ns + s)) + sh[q];
    }
    __device__ __forceinline__ void st(int d, int s, int q, float v) const
    {
        if constexpr (std::is_same<T, float>::value) PopIO<T>::st(f + (d * ns + s), v);
        else PopIO<T>::st(f + (d * ns + s), v - sh[q]);
    }
    // two consecutive slots from an even s, through the thread's own shared memory
    __device__ __forceinline__ void fetch2(int d, int s, T *buf) const { async_copy<2 * sizeof(T)>(buf, f + (d * ns + s)); }
    __device__ __forceinline__ void fetched2(int q, const T *buf, float v[2]) const
    {
        const float2 a = pop_ld2(buf);
        v[0] = a.x; v[1] = a.y;
        if constexpr (!std::is_same<T, float>::value) { v[0] += sh[q]; v[1] += sh[q]; }
    }
    __device__ __forceinline__ void st2(int d, int s, int q, float a, float b) const
    {
        if constexpr (std::is_same<T, float>::value) pop_st2(f + (d * ns + s), a, b);
        else pop_st2(f + (d * ns + s), a - sh[q], b - sh[q]);
    }
};

// outlet buffer index of direction 2, 6 or 8
__device__ __forceinline__ int obuf_m(int q) { return q == 2 ? 0 : (q == 6 ? 1 : 2); }

// Post-collision populations o of an active fluid cell into the layout the next step of
// the level reads: an even step (ODD false) keeps them in the cell's own slots, an odd
// step sends each to the downstream cell, with the level-0 box edges (specular reflection
// at the symmetry planes, nothing across the inlet and the outlet).  nbs / present: slots
// at offsets +c_q and the mask of the present ones.  Boundary nodes, outlet columns and
// band cells also fill their side buffers (the explosion is done by the caller).
template <typename T, bool ODD>
__device__ __forceinline__ void put_post(const Lat<T> &F, const StepConsts &k, int slot, const int nbs[9],
                                         unsigned present, bool edge, int gi, int gj, const float o[9])
{
    if (!ODD) {
#pragma unroll
        for (int q = 0; q < 9; q++) F.st(oppq(q), slot, q, o[q]);
    } else if (!edge) {
        F.st(0, slot, 0, o[0]);
#pragma unroll
        for (int q = 1; q < 9; q++)
            if (present >> q & 1) F.st(q, nbs[q], q, o[q]);
    } else {
        F.st(0, slot, 0, o[0]);
#pragma unroll
        for (int q = 1; q < 9; q++) {
            const int di = gi + cxq(q), dj = gj + cyq(q);
            if (di < 0 || di >= k.nx0) continue;                       // across the inlet or the outlet
            if (dj >= 0 && dj < k.ny0) F.st(q, slot0(k, di, dj), q, o[q]);
            else F.st(mirror_y(q), slot0(k, di, gj), mirror_y(q), o[q]);  // reflected at the plane
        }
    }
}

// Outlet side buffer (parity par): the populations 2, 6, 8 of the outlet columns N-1 and N-2
// (flags FL_OUTLET, FL_OUTLET2) at row gj.
__device__ __forceinline__ void put_obuf(const StepConsts &k, int par, uint32_t fl, int gj, const float o[9])
{
    float *ob = k.obuf + par * (6 * k.ny0) + ((fl & FL_OUTLET) ? 0 : 3 * k.ny0);
    ob[gj] = o[2]; ob[k.ny0 + gj] = o[6]; ob[2 * k.ny0 + gj] = o[8];
}

// Explosion (Rohde, Sec 2.1) of band cell (t, lx, ly) with post-collision populations o: they
// become those of its four ghost children, written where the fine level's next even sub-step
// reads them (slot (g + c_q, q) for child g).  Children that are solid or have no tile relay
// nothing, so their share of the next coalescence is this value too.
//
// The targets of all four children lie in the 4 x 4 cells around them.  Their slots are static:
// tgt holds, per row cy0 - 1 .. cy0 + 2 of the cells (cx0 .. cx0 + 1, cy0 .. cy0 + 1), the slots
// of cx0 - 1, of cx0 (and cx0 + 1, the next one) and of cx0 + 2, -1 where there is no tile, so that
// the stores wait for no table; the two children of a row share one 64-bit store where c_x = 0.
struct BandTargets {
    int4 row[4];
};

__device__ __forceinline__ BandTargets band_targets(const LevelView &P, int b)
{
    BandTargets t;
#pragma unroll
    for (int a = 0; a < 4; a++) t.row[a] = __ldg(P.band_tgt + 4 * b + a);
    return t;
}

template <typename T>
__device__ __forceinline__ void explode_band(const LevelView &P, const LevelView &F, const StepConsts &k, uint32_t fl, int b,
                                             const BandTargets &tgt, const float o[9], int *status = nullptr)
{
    float *eb = P.ebuf + b * 9;
#pragma unroll
    for (int q = 0; q < 9; q++) eb[q] = o[q];
    const uint32_t sch = fl >> FL_SCH_SHIFT;
#pragma unroll
    for (int m = 0; m < 4; m++) {
        if (sch >> m & 1) {
            float *gb = P.gbuf + (4 * b + m) * 9;
#pragma unroll
            for (int q = 0; q < 9; q++) gb[q] = o[q];
        }
    }
    const Lat<T> LF{static_cast<T *>(F.f), F.ns, k.pshift};
#pragma unroll
    for (int q = 0; q < 9; q++) {
#pragma unroll
        for (int my = 0; my < 2; my++) {
            const int4 t = tgt.row[my + cyq(q) + 1];
            const int in = t.y < 0 ? -1 : checked_index(t.y, F.ns - 1, status);
            if (cxq(q) == 0) {
                if (in >= 0) LF.st2(q, in, q, o[q], o[q]);
            } else {
                // the children at cx0 and cx0 + 1 write to cx0 + c_x and cx0 + 1 + c_x
                const int far = cxq(q) > 0 ? t.z : t.x, out = far < 0 ? -1 : checked_index(far, F.ns, status);
                if (in >= 0) LF.st(q, cxq(q) > 0 ? in + 1 : in, q, o[q]);
                if (out >= 0) LF.st(q, out, q, o[q]);
            }
        }
    }
}

// Whether a cell's aux word is used by the level step: ghosts, boundary nodes, band cells
// and coalescing cells.
__device__ __forceinline__ bool uses_aux(uint32_t fl)
{
    return (fl & FL_KIND_MASK) == KIND_GHOST || (fl & (FL_BNODE | FL_BAND | (0xFFu << FL_COAL_SHIFT)));
}

// ------------------------------------------------------------------ work of a warp
// The static part of a warp's work, read before the wait for the preceding kernel.  The work list
// holds the general 16 x 2-cell blocks (each with boundary nodes twice: its wall warp, then its
// partner), then the plain ones.  A PLAIN launch takes the latter two to a warp (plain_warp),
// any other one to a warp as it takes the general ones.
struct GeneralWork {
    int t;              // tile
    bool wall;          // one of a pair of warps
    int lx, ly;         // the lane's cell
    uint32_t fl;
    int ax;
    int s[9];           // own slot and those at offsets +c_q (the own one where there is no tile)
    unsigned present;   // mask of the neighbours that have a tile
    int ps;             // with a restriction: slot of the cell's parent, or -1
};

struct PlainWork {
    int e;              // tile * 8 + block of the tile
    int tv, th0, thv;   // tiles across the lane's vertical / horizontal / both tile edges, its own
                        // where it has none
};

// warps that a launch over a level takes
__host__ __device__ __forceinline__ int level_warps(const LevelView &P, bool plain)
{
    return P.n_gen_warps + (plain ? P.n_plain / 2 : P.n_plain);
}

__device__ __forceinline__ GeneralWork general_work(const LevelView &P, const LevelView &C, const LevelStep &ls, int w, int lane,
                                                    int *nb3)
{
    GeneralWork W;
    const int e = checked_index(__ldg(P.work + w), 8 * P.ntiles, ls.status), t = e >> 3;
    W.t = t;
    W.wall = w < P.n_pair_warps;
    cell_of_thread((e & 7) * 32 + lane, W.lx, W.ly);
    if (lane < 9) nb3[lane] = P.nbr[t * 9 + dir_of3(lane)];
    const int slot = t * LBM_TILE + W.ly * LBM_TX + W.lx;
    W.fl = __ldg(P.flags + slot);
    W.ax = uses_aux(W.fl) ? __ldg(P.aux + slot) : -1;
    __syncwarp();
    W.present = neighbours(nb3, W.lx, W.ly, slot, W.s);
#ifdef LBM_BOUNDS_CHECK
#pragma unroll
    for (int q = 1; q < 9; q++) W.s[q] = checked_index(W.s[q], P.ns, ls.status);
#endif
    W.ps = -1;
    if (ls.restrict_up) {
        const int pt = __ldg(P.parent + t);
        const int px = (__ldg(P.tile_x + t) & 1) * (LBM_TX / 2) + (W.lx >> 1);
        const int py = (__ldg(P.tile_y + t) & 1) * (LBM_TY / 2) + (W.ly >> 1);
        if (pt >= 0) W.ps = checked_index(pt, C.ntiles, ls.status) * LBM_TILE + py * LBM_TX + px;
    }
    return W;
}

__device__ __forceinline__ PlainWork plain_work(const LevelView &P, const LevelStep &ls, int w, int lane)
{
    PlainWork W;
    W.e = checked_index(__ldg(P.work + P.n_gen_warps + 2 * (w - P.n_gen_warps) + (lane >> 4)), 8 * P.ntiles, ls.status);
    const int t = W.e >> 3, li = lane & 15;
    const int lx = (W.e & 1) * 16 + (li & 7) * 2, ly = ((W.e >> 1) & 3) * 2 + (li >> 3);
    const int sx = lx == 0 ? 0 : (lx == LBM_TX - 2 ? 2 : 1), sy = ly == 0 ? 0 : (ly == LBM_TY - 1 ? 2 : 1);
    const int *nb = P.nbr + t * 9;
    W.tv = sy == 1 ? t : __ldg(nb + dir_of3(sy * 3 + 1));
    W.th0 = sx == 1 ? t : __ldg(nb + dir_of3(3 + sx));
    W.thv = sx == 1 ? W.tv : (sy == 1 ? W.th0 : __ldg(nb + dir_of3(sy * 3 + sx)));
    return W;
}

// ------------------------------------------------------------------ wall warps
// A block of cells with boundary nodes takes two warps: this one evaluates the wall function of
// the block's records (Sec 2.3 steps 1-5) while its partner (general_warp) loads and updates the
// cells; the results pass through shared memory, indexed by the cell's lane.  The records are
// packed: up to 8 take four lanes each, up to 16 two, which share the 16-entry stencil's gather
// (a row of the stencil a lane) and then evaluate the same record.
struct WallPair {
    float4 res[32];     // per cell lane: rho_W - 1, u_W, chi_B
    int rec[32];        // packed records and the lanes of their cells
    int cell[32];
};

// The pair's named barrier (1 or 2; both warps of a pair, 64 threads).  The barrier's number is a
// constant in each branch: with a number from a register the block would reserve all 16 barriers,
// which leaves room for four blocks per SM (the c/4096 workload's finest level: 17.7 / 21.2 us for
// its even / odd step that way, 13.8 / 16.5 us this way).
// Both instructions are the aligned forms, which all lanes of a warp must execute together, and
// they order memory between the warps only for what each lane wrote before.  What precedes them
// branches per lane (the Newton iteration's length, the lanes that hold a result), so each first
// brings its warp's lanes together.
__device__ __forceinline__ void pair_arrive(int pair)
{
    __syncwarp();
    if (pair == 0) asm volatile("bar.arrive 1, 64;" ::: "memory");
    else asm volatile("bar.arrive 2, 64;" ::: "memory");
}
__device__ __forceinline__ void pair_wait(int pair)
{
    __syncwarp();
    if (pair == 0) asm volatile("bar.sync 1, 64;" ::: "memory");
    else asm volatile("bar.sync 2, 64;" ::: "memory");
}

// A boundary node's weights q / (1 + q) of the wall fractions and the mask of directions q whose node
// B + c_q is active fluid (eq 27), read before the wait.
struct CutLinks {
    float v[9];
    uint32_t nf;
};

// Eq 27 for one cut direction of wall fraction q: gin the population that arrives along the opposite
// one, fo and f the cell's own last post-collision ones along it and along the direction, mom the
// wall's momentum term, v = q / (1 + q).  The quotient ((1 - q) gin + q fo + mom + q f) / (1 + q) is
// gin + mom + v (fo + f - 2 gin - mom): the roundings act on small differences, and no division
// follows the wall warp's results.  Error against 64 bits, in the populations' size: 1.4e-8 rms and
// 0.8e-7 at most; with weights 1 / (1 + q) and q / (1 + q) rounded to FP32 2.7e-8 and 1.8e-7, and
// dividing the whole sum 3.9e-8 and 2.9e-7.
__device__ __forceinline__ float yu_link(float v, float gin, float fo, float f, float mom)
{
    return gin + (mom + v * ((fo - gin) + (f - gin) - mom));
}

struct WallStatic {
    int n, sh, r, cell;           // records, lanes a record as a shift, the lane's record and its cell's lane
    int4 sl;                      // the lane's first stencil row: slots and weights
    float4 wr, wu;
    float nx, ny, dwb;
};

// the static part, before the wait for the preceding kernel (bnode: the lane's cell is a
// boundary node, ax its record)
__device__ __forceinline__ WallStatic wall_static(const RecView &R, WallPair &S, bool bnode, int ax, int lane, int *status)
{
    WallStatic W;
    const unsigned m = __ballot_sync(0xffffffffu, bnode);
    if (bnode) {
        const int j = __popc(m & ((1u << lane) - 1u));
        S.rec[j] = checked_index(ax, R.n, status);
        S.cell[j] = lane;
    }
    __syncwarp();
    W.n = __popc(m);
    W.sh = W.n <= 8 ? 2 : (W.n <= 16 ? 1 : 0);
    const int j = lane >> W.sh;
    const bool have = j < W.n;
    W.r = S.rec[have ? j : 0];
    W.cell = have ? S.cell[j] : -1;
    const int m4 = lane & ((1 << W.sh) - 1);
    W.sl = __ldg(reinterpret_cast<const int4 *>(R.st_slot + W.r * 16) + m4);
    W.wr = __ldg(reinterpret_cast<const float4 *>(R.st_wr + W.r * 16) + m4);
    W.wu = __ldg(reinterpret_cast<const float4 *>(R.st_wu + W.r * 16) + m4);
    W.nx = __ldg(R.nx + W.r); W.ny = __ldg(R.ny + W.r); W.dwb = __ldg(R.dwb + W.r);
    return W;
}

__device__ __forceinline__ void wall_warp(const LevelView &P, const RecView &R, const StepConsts &k, const LevelStep &ls,
                                          const WallStatic &W, WallPair &S, int lane)
{
    const int nl = 1 << W.sh, m0 = lane & (nl - 1);
    const float start = R.utau_start[W.r];
    float drR = 0.f, uR = 0.f, vR = 0.f;
    wall_gather(P, ls.p, W.sl, W.wr, W.wu, drR, uR, vR, ls.status);
    for (int m4 = m0 + nl; m4 < 4; m4 += nl)
        wall_gather(P, ls.p, __ldg(reinterpret_cast<const int4 *>(R.st_slot + W.r * 16) + m4),
                    __ldg(reinterpret_cast<const float4 *>(R.st_wr + W.r * 16) + m4),
                    __ldg(reinterpret_cast<const float4 *>(R.st_wu + W.r * 16) + m4), drR, uR, vR, ls.status);
    for (int d = 1; d < nl; d <<= 1) {
        drR += __shfl_xor_sync(0xffffffffu, drR, d); uR += __shfl_xor_sync(0xffffffffu, uR, d);
        vR += __shfl_xor_sync(0xffffffffu, vR, d);
    }
    const WallState w = wall_point(P, R, k, W.r, W.nx, W.ny, W.dwb, start, uR, vR);
    if (W.cell >= 0 && m0 == 0) {
        if (k.wall_model < 2) R.utau_start[W.r] = w.utau;
        S.res[W.cell] = make_float4(drR, w.uWx, w.uWy, w.chiB);
    }
}

// One 16 x 2-cell warp of the fused level step, one cell a lane, for blocks of cells with
// anything besides plain active cells in them: every kind of cell, level-0 edges, walls,
// interfaces.
//
// A launch of a small level is one such warp's latency (a round trip to L2 is about 0.5 us, and a
// warp alone issues an instruction every three to four cycles), so the loads come first and in as
// few dependent rounds as the data allows: flag words, neighbour tiles, cut links and the wall
// records' tables are read before the wait for the preceding kernel; the arriving populations,
// the side buffer's values (a ghost's kept ones, a boundary node's last ones) and the SA stencil
// go out together, for every lane and whatever its kind; the coalescence buffers follow as one
// round instead of one per direction, and the wall function runs in a warp of its own (wall_warp).
// c/256 airfoil: the finest level's launch 9.7 / 12.9 us (even / odd) with the code of one cell a
// thread and the boundary nodes' work in line, 2.8 / 3.2 us this way; level 4 (interfaces on both
// sides) 4.9 / 6.6 us, then 3.3 / 4.6 with neighbour slots, parents and the explosion's targets
// found after the wait, now 2.6 / 3.3 us.
template <int KIND, typename T, bool ODD, bool PLAIN, bool EDGE>
__device__ __forceinline__ void general_warp(const LevelView &P, const LevelView &F, const LevelView &C, const RecView &R,
                                             const StepConsts &k, const LevelStep &ls, const Lat<T> &L, const GeneralWork &W,
                                             int lane, const WallPair *wp, int pair, const CutLinks &cut)
{
    constexpr bool CHILD = KIND == 1, WALL = KIND == 2;
    const int *nbs = W.s, slot = W.s[0], t = W.t, lx = W.lx, ly = W.ly;
    const unsigned present = W.present;
    const uint32_t fl = W.fl;
    int ax = W.ax;
    const uint32_t kind = fl & FL_KIND_MASK;
    const bool fluid = !(fl & FL_SOLID);
    const bool act = kind == KIND_ACTIVE && fluid, ghost = kind == KIND_GHOST && fluid;
    const int p = ls.p;
    float n_dr = 0.f, n_ux = 0.f, n_uy = 0.f, n_chi = 0.f;

    const bool edge = EDGE && act && (fl & (FL_INLET | FL_OUTLET | FL_BOTTOM | FL_TOP));
    const bool bnode = WALL && act && (fl & FL_BNODE);
    // ---- streaming (eq 1): the populations arriving at the cell.  (Where no upstream tile
    // exists the own slot is read and the value replaced below.)
    float g[9];
    g[0] = L.ld(0, slot, 0);
#pragma unroll
    for (int q = 1; q < 9; q++) g[q] = ODD ? L.ld(oppq(q), nbs[oppq(q)], q) : L.ld(q, slot, q);
    // side buffer of the cell: a ghost's parent's exploded populations, or a boundary
    // node's last post-collision ones
    float x[9];
    int r = -1;
    {
        const float *sb = nullptr;
        if (ghost) {
            ax = checked_index(ax, 4 * C.n_band, ls.status);
            sb = C.ebuf + (ax >> 2) * 9;
        } else if (bnode) {
            r = checked_index(ax, R.n, ls.status);
            sb = R.fpost + r * 9;
        }
#pragma unroll
        for (int q = 0; q < 9; q++) x[q] = sb ? sb[q] : 0.0f;
    }
    const bool band = CHILD && act && (fl & FL_BAND);
    if (CHILD && act && (fl & (FL_BAND | (0xFFu << FL_COAL_SHIFT)))) ax = checked_index(ax, P.n_band, ls.status);
    // the explosion's targets: with the first round of loads where the registers allow it (launches
    // without plain warps), else behind the SA-neg update
    BandTargets tgt = {};
    if (!PLAIN && band) tgt = band_targets(P, ax);
    Stencil S;
    const bool sa = k.turbulence != 0 && __any_sync(0xffffffffu, act);
    if (sa) {
        const float *xc = P.chi[p], *xu = P.ux[p], *xv = P.uy[p];
#pragma unroll
        for (int q = 0; q < 9; q++) {
            S.chi[q] = xc[nbs[q]]; S.ux[q] = xu[nbs[q]]; S.uy[q] = xv[nbs[q]];
        }
    }
    float id2 = sa ? __ldg(P.inv_d2 + slot) : 0.0f;
    // (keeps the compiler from moving the stencil's loads down to their use, behind the branches
    // below and the loads that they wait for)
    asm volatile("" ::: "memory");
    int gi = 0, gj = 0;
    if (edge) {
        gi = P.tile_x[t] * LBM_TX + lx; gj = P.tile_y[t] * LBM_TY + ly;
        if (sa && !bnode) {
            const int ic = (fl & FL_OUTLET) ? k.nx0 - 2 : gi;     // outlet: copy of its neighbour
            gather0(P.chi[p], P.ux[p], P.uy[p], k, ic, gj, S);
            id2 = P.inv_d2[slot0(k, ic, gj)];
        }
        if (ODD) {
            // level-0 box edge: in-box pulls and the symmetry planes' reflections
#pragma unroll
            for (int q = 1; q < 9; q++) {
                const int si = gi - cxq(q), sj = gj - cyq(q);
                const bool xin = si >= 0 && si < k.nx0, yin = sj >= 0 && sj < k.ny0;
                if (xin && yin) g[q] = L.ld(oppq(q), slot0(k, si, sj), q);
                else if (xin) g[q] = L.ld(oppq(mirror_y(q)), slot0(k, si, gj), mirror_y(q));
                else g[q] = 0.0f;
            }
        }
    }
    if (CHILD && (fl & (0xFFu << FL_COAL_SHIFT)) && act) {
        // coalescence: mean of what the four ghost children pulled in the fine level's odd sub-step
        const float4 *gb = reinterpret_cast<const float4 *>(P.gbuf + ax * 36);
        float c[36];                                      // child m's population q at 9 m + q
#pragma unroll
        for (int i = 0; i < 9; i++) {
            const float4 v = gb[i];
            c[4 * i] = v.x; c[4 * i + 1] = v.y; c[4 * i + 2] = v.z; c[4 * i + 3] = v.w;
        }
#pragma unroll
        for (int q = 1; q < 9; q++)
            if (fl & (1u << (FL_COAL_SHIFT + q - 1))) g[q] = 0.25f * (c[q] + c[9 + q] + c[18 + q] + c[27 + q]);
    }
    // ---- SA-neg update of chi (Sec 2.2), fields at time t
    float chin = 0.0f;
    if (act) {
        if (!sa) chin = P.chi[p][slot];
        else if (edge && (fl & FL_INLET)) chin = k.chi_inf;
        else chin = sa_update(S, id2, P.nu, k.sa_convection);
    }
    if (PLAIN && band) tgt = band_targets(P, ax);
    // ---- wall function of the boundary nodes (Sec 2.3), fields at time t, from the partner warp
    // (all lanes wait, whatever their cells)
    float drW = 0.f, uWx = 0.f, uWy = 0.f;
    if (WALL && wp) {
        pair_wait(pair);
        if (bnode) {
            const float4 w = wp->res[lane];
            drW = w.x; uWx = w.y; uWy = w.z;
            if (sa) chin = w.w;                                     // Dirichlet nu_t~_B (Sec 2.2)
        }
    }
    if (ghost) {
        // ghosts are streamed (relayed), never collided.  Where the upstream cell is not fluid
        // the ghost keeps its own value, the parent's exploded one.  Even sub-step: the
        // arriving populations stay in the cell, moved to the slots an odd step reads; odd
        // sub-step: the pulled populations go to the parent's coalescence buffer.
        const uint32_t keep = fl >> FL_KEEP_SHIFT;
#pragma unroll
        for (int q = 1; q < 9; q++)
            if ((keep >> (q - 1) & 1) || (ODD && !(present >> oppq(q) & 1))) g[q] = x[q];
        if (!ODD) {
#pragma unroll
            for (int q = 0; q < 9; q++) L.st(oppq(q), slot, q, g[q]);
        } else {
            float *gb = C.gbuf + ax * 9;
#pragma unroll
            for (int q = 0; q < 9; q++) gb[q] = g[q];
        }
    } else if (act) {
        if (sa) P.chi[p ^ 1][slot] = chin;
        if (WALL && bnode && (fl & (0xFFu << FL_CUT_SHIFT))) {
            // Yu's interpolated bounce-back with the slip velocity of the wall record (eq 27): the
            // next fluid node's f*_qo arrives at B as its own f_qo; f*_q(B) and f*_qo(B) of the last
            // step come from the record's buffer
            float gin[9];
#pragma unroll
            for (int q = 0; q < 9; q++) gin[q] = g[q];
#pragma unroll
            for (int q = 1; q < 9; q++) {
                const int qo = oppq(q);
                const float mom = 6.0f * wq(q) * (1.0f + drW) * (cxq(q) * uWx + cyq(q) * uWy);
                const float yu = yu_link(cut.v[q], gin[qo], x[qo], x[q], mom);
                const float half = x[qo] + mom;           // half-way form, eq 24
                if (fl & (1u << (FL_CUT_SHIFT + q - 1))) g[q] = (cut.nf >> q & 1) ? yu : half;
            }
        }
        if (edge) {
            if (gi == 0) {
                // Zou-He velocity inlet (Sec 3.1.1)
                const float U = k.U;
                const float Sg = g[0] + g[3] + g[4] + 2.0f * (g[2] + g[6] + g[8]);   // sum of w over these is 1
                const float rho = (1.0f + Sg) / (1.0f - U);
                g[1] = g[2] + (2.0f / 3.0f) * rho * U;
                g[5] = g[6] - 0.5f * (g[3] - g[4]) + rho * U * (1.0f / 6.0f);
                g[7] = g[8] + 0.5f * (g[3] - g[4]) + rho * U * (1.0f / 6.0f);
            }
            if (gi == k.nx0 - 1) {
                // outlet, for the directions 2, 6, 8 entering from outside, on the post-stream
                // values of the columns N-2 and N-3 (the post-collision values of the columns
                // N-1 and N-2 one row up or down, or reflected at a symmetry plane):
                // Yu's linear extrapolation 2 g_q(N-2) - g_q(N-3), or the zero-gradient copy g_q(N-2)
                const float *ob = k.obuf + p * (6 * k.ny0);
#pragma unroll
                for (int m = 0; m < 3; m++) {
                    const int q = m == 0 ? 2 : (m == 1 ? 6 : 8);
                    const int sj = gj - cyq(q);
                    const bool yin = sj >= 0 && sj < k.ny0;
                    const int ms = obuf_m(yin ? q : mirror_y(q)), js = yin ? sj : gj;
                    const float g2 = ob[ms * k.ny0 + js];
                    g[q] = k.outlet == 0 ? 2.0f * g2 - ob[(3 + ms) * k.ny0 + js] : g2;
                }
            }
        }
        // ---- macroscopic fields (eq 3) and central-moment collision (eqs 5-11)
        const float drho = g[0] + g[1] + g[2] + g[3] + g[4] + g[5] + g[6] + g[7] + g[8];
        const float jx = g[1] - g[2] + g[5] - g[6] + g[7] - g[8];
        const float jy = g[3] - g[4] + g[5] - g[6] - g[7] + g[8];
        const float irho = __fdividef(1.0f, 1.0f + drho);
        const float ux = jx * irho, uy = jy * irho;
        P.drho[p ^ 1][slot] = drho; P.ux[p ^ 1][slot] = ux; P.uy[p ^ 1][slot] = uy;
        float o[9];
        collide_cm(g, drho, jx, jy, ux, uy, delta_of(P.nu, chin, k.turbulence), o);
        put_post<T, ODD>(L, k, slot, nbs, present, edge, gi, gj, o);
        if (bnode) {
            float *fp = R.fpost + r * 9;
#pragma unroll
            for (int q = 0; q < 9; q++) fp[q] = o[q];
        }
        if (EDGE && (fl & (FL_OUTLET | FL_OUTLET2)))
            put_obuf(k, p ^ 1, fl, P.tile_y[t] * LBM_TY + ly, o);
        if (band) explode_band<T>(P, F, k, fl, ax, tgt, o, ls.status);
        n_dr = drho; n_ux = ux; n_uy = uy; n_chi = chin;
    }

    if (ls.restrict_up) {
        // restriction into the covered parents (their children are this level's active
        // cells): rho and chi are the means over the fluid children, u is mass-weighted
        // (Rohde transfers, Sec 2.1).  A 2 x 2 group lies inside the warp, lanes l, l+1, l+16,
        // l+17: sum over (l, l+1) then over (l, l+16)
        const float rr = act ? 1.0f + n_dr : 0.0f;
        float a0 = act ? n_dr : 0.0f, a1 = rr, a2 = rr * n_ux, a3 = rr * n_uy, a4 = act ? n_chi : 0.0f;
        float a5 = act ? 1.0f : 0.0f;
#pragma unroll
        for (int d = 1; d <= 16; d <<= 4) {
            a0 += __shfl_down_sync(0xffffffffu, a0, d); a1 += __shfl_down_sync(0xffffffffu, a1, d);
            a2 += __shfl_down_sync(0xffffffffu, a2, d); a3 += __shfl_down_sync(0xffffffffu, a3, d);
            a4 += __shfl_down_sync(0xffffffffu, a4, d); a5 += __shfl_down_sync(0xffffffffu, a5, d);
        }
        if (!(lane & 1) && lane < 16 && kind == KIND_ACTIVE) {
            const int n = (int)a5, ps = W.ps, q1 = ls.pp ^ 1;
            if (ps >= 0 && n > 0) {
                C.drho[q1][ps] = a0 / n; C.ux[q1][ps] = a2 / a1; C.uy[q1][ps] = a3 / a1;
                C.chi[q1][ps] = a4 / n;
            }
        }
    }
}

__device__ __forceinline__ void ld2(const float *a, float v[2])
{
    const float2 m = *reinterpret_cast<const float2 *>(a);
    v[0] = m.x; v[1] = m.y;
}
__device__ __forceinline__ void st2(float *a, const float v[2]) { *reinterpret_cast<float2 *>(a) = make_float2(v[0], v[1]); }

// Row of four values around a lane's two cells: the cell to the left, the two, the one to the right.
__device__ __forceinline__ void row4(const float *a, int left, int mid, int right, float v[4])
{
    v[0] = a[left];
    ld2(a + mid, v + 1);
    v[3] = a[right];
}

// One warp over two plain 16 x 2-cell blocks (every cell active, none with a wall, interface or
// box edge, all neighbour tiles present), sixteen lanes a block, two cells of a row a lane.  No
// flag word is read and nothing branches on a cell.  Fields and populations move as pairs, and a
// stencil row costs two more scalar loads instead of four: 422 (even) and 446 (odd) warp instructions
// for 32 cells with SA-neg where one cell a lane took 641 and 751.  The populations come through the
// thread's own shared memory (buf, asynchronous copies): they are in flight during the SA-neg update
// without holding registers, so one round of memory latency is exposed instead of two.
// 2048^2 level, SA-neg, FP32: 126.5 -> 91 us a step (5.0 TB/s of the method's 108 B a cell); 3008 x
// 2792, laminar: 185 -> 128 us (5.8 TB/s of 88 B); 1536 x 2048, SA-neg, BF16: 100 -> 66.6 us.
// Four cells a lane (half as many stencil loads) needs 96 registers or spills, keeps a third fewer
// cells in flight and came out at 92.6, 133 and 66 us; without the copies through shared memory
// two cells a lane at 96 registers took 114, 165 and 82 us.
template <typename T, bool ODD>
__device__ __forceinline__ void plain_warp(const LevelView &P, const LevelView &C, const StepConsts &k, const LevelStep &ls,
                                           const Lat<T> &L, const PlainWork &W, int lane, T *buf)
{
    const int t = W.e >> 3, li = lane & 15;
    const int lx = (W.e & 1) * 16 + (li & 7) * 2, ly = ((W.e >> 1) & 3) * 2 + (li >> 3);
    const int p = ls.p;
    // slots of the lane's first cell, one row down (0), its own (1), one row up (2), and of the
    // cells left and right of the two in those rows (found here and not before the wait: nine
    // registers less to hold there, a 2048^2 level takes 87 us a step instead of 94)
    int mid[3], lf[3], rt[3];
    {
        const bool wl = lx == 0, wr = lx == LBM_TX - 2;
#pragma unroll
        for (int a = 0; a < 3; a++) {
            const int y = ly + a - 1;
            const bool over = y < 0 || y >= LBM_TY;
            const int row = (y & (LBM_TY - 1)) * LBM_TX;
            mid[a] = (over ? W.tv : t) * LBM_TILE + row + lx;
            const int ts = (over ? W.thv : W.th0) * LBM_TILE + row;
            lf[a] = wl ? ts + LBM_TX - 1 : mid[a] - 1;
            rt[a] = wr ? ts : mid[a] + 2;
#ifdef LBM_BOUNDS_CHECK
            mid[a] = checked_index(mid[a], P.ns - 1, ls.status) & ~1;
            lf[a] = checked_index(lf[a], P.ns, ls.status); rt[a] = checked_index(rt[a], P.ns, ls.status);
#endif
        }
    }
    const int slot = mid[1];
    // ---- streaming (eq 1): fetch the populations arriving at the cells; in odd steps those of the
    // upstream rows y - c_y from the opposite planes
    buf += lane * 2;
#pragma unroll
    for (int q = 0; q < 9; q++) {
        if (!ODD) L.fetch2(q, slot, buf + q * 64);
        else L.fetch2(oppq(q), mid[1 - cyq(q)], buf + q * 64);
    }
    // ---- SA-neg update of chi (Sec 2.2), fields at time t
    float chin[2];
    if (k.turbulence) {
        float x[3][4], um[4], up[4], vm[4], v0[4], vp[4], vort[2], u0[2], id2[2];
        const float *pc = P.chi[p], *pu = P.ux[p], *pv = P.uy[p];
#pragma unroll
        for (int a = 0; a < 3; a++) row4(pc, lf[a], mid[a], rt[a], x[a]);
        row4(pu, lf[0], mid[0], rt[0], um); row4(pu, lf[2], mid[2], rt[2], up);
        ld2(pu + slot, u0);
        row4(pv, lf[0], mid[0], rt[0], vm); row4(pv, lf[1], mid[1], rt[1], v0); row4(pv, lf[2], mid[2], rt[2], vp);
        ld2(P.inv_d2 + slot, id2);
        const float lo = fminf(fminf(fminf(x[1][0], x[1][1]), fminf(x[1][2], x[1][3])),
                               fminf(fminf(x[0][1], x[0][2]), fminf(x[2][1], x[2][2])));
#pragma unroll
        for (int c = 0; c < 2; c++) {
            // LSQ gradients over the full neighbourhood (lsq_grad): du/dy and dv/dx
            const float dudy = ((up[c + 1] - um[c + 1]) + (up[c + 2] - um[c]) + (up[c] - um[c + 2])) * (1.0f / 6.0f);
            const float dvdx = ((v0[c + 2] - v0[c]) + (vp[c + 2] - vm[c]) + (vm[c + 2] - vp[c])) * (1.0f / 6.0f);
            vort[c] = fabsf(dvdx - dudy);
        }
#pragma unroll
        for (int c = 0; c < 2; c++) {
            const float s[9] = {x[1][c + 1], x[1][c + 2], x[1][c], x[2][c + 1], x[0][c + 1],
                                x[2][c + 2], x[0][c], x[0][c + 2], x[2][c]};
            chin[c] = lo >= 0.0f ? sa_point<true>(s, u0[c], v0[c + 1], vort[c], id2[c], P.nu, k.sa_convection)
                                 : sa_point<false>(s, u0[c], v0[c + 1], vort[c], id2[c], P.nu, k.sa_convection);
        }
        st2(P.chi[p ^ 1] + slot, chin);
    } else {
        // laminar: chi takes no part in the step, but the covered parents' is restricted below
        chin[0] = chin[1] = 0.0f;
        if (ls.restrict_up) ld2(P.chi[p] + slot, chin);
    }
    // odd steps: the cell beside the two where c_x != 0 (mostly in a line that a neighbour lane has
    // fetched by now; loaded here so as not to hold six registers through the SA-neg update)
    float side[9];
    if (ODD) {
#pragma unroll
        for (int q = 1; q < 9; q++)
            if (cxq(q) != 0) side[q] = L.ld(oppq(q), cxq(q) > 0 ? lf[1 - cyq(q)] : rt[1 - cyq(q)], q);
    }
    async_wait();
    float g[9][2];
#pragma unroll
    for (int q = 0; q < 9; q++) {
        float v[2];
        L.fetched2(q, buf + q * 64, v);
        g[q][0] = ODD && cxq(q) > 0 ? side[q] : (ODD && cxq(q) < 0 ? v[1] : v[0]);
        g[q][1] = ODD && cxq(q) < 0 ? side[q] : (ODD && cxq(q) > 0 ? v[0] : v[1]);
    }
    // ---- macroscopic fields (eq 3) and central-moment collision (eqs 5-11)
    float dr[2], ux[2], uy[2];
#pragma unroll
    for (int c = 0; c < 2; c++) {
        const float gc[9] = {g[0][c], g[1][c], g[2][c], g[3][c], g[4][c], g[5][c], g[6][c], g[7][c], g[8][c]};
        dr[c] = gc[0] + gc[1] + gc[2] + gc[3] + gc[4] + gc[5] + gc[6] + gc[7] + gc[8];
        const float jx = gc[1] - gc[2] + gc[5] - gc[6] + gc[7] - gc[8];
        const float jy = gc[3] - gc[4] + gc[5] - gc[6] - gc[7] + gc[8];
        const float irho = __fdividef(1.0f, 1.0f + dr[c]);
        ux[c] = jx * irho; uy[c] = jy * irho;
        float o[9];
        collide_cm(gc, dr[c], jx, jy, ux[c], uy[c], delta_of(P.nu, chin[c], k.turbulence), o);
#pragma unroll
        for (int q = 0; q < 9; q++) g[q][c] = o[q];
    }
    st2(P.drho[p ^ 1] + slot, dr);
    st2(P.ux[p ^ 1] + slot, ux);
    st2(P.uy[p ^ 1] + slot, uy);
#pragma unroll
    for (int q = 0; q < 9; q++) {
        const int a = 1 + cyq(q);
        if (!ODD) L.st2(oppq(q), slot, q, g[q][0], g[q][1]);
        else if (cxq(q) == 0) L.st2(q, mid[a], q, g[q][0], g[q][1]);
        else if (cxq(q) > 0) { L.st(q, mid[a] + 1, q, g[q][0]); L.st(q, rt[a], q, g[q][1]); }
        else { L.st(q, lf[a], q, g[q][0]); L.st(q, mid[a], q, g[q][1]); }
    }
    if (ls.restrict_up) {
        // restriction (as in general_warp): the lane's pair and that of the lane one row up
        const float r0 = 1.0f + dr[0], r1 = 1.0f + dr[1];
        float a0 = dr[0] + dr[1], a1 = r0 + r1, a2 = r0 * ux[0] + r1 * ux[1], a3 = r0 * uy[0] + r1 * uy[1];
        float a4 = chin[0] + chin[1];
        a0 += __shfl_down_sync(0xffffffffu, a0, 8); a1 += __shfl_down_sync(0xffffffffu, a1, 8);
        a2 += __shfl_down_sync(0xffffffffu, a2, 8); a3 += __shfl_down_sync(0xffffffffu, a3, 8);
        a4 += __shfl_down_sync(0xffffffffu, a4, 8);
        int pt = li < 8 ? P.parent[t] : -1;
#ifdef LBM_BOUNDS_CHECK
        if (pt >= 0) pt = checked_index(pt, C.ntiles, ls.status);
#endif
        if (pt >= 0) {
            const int px = (P.tile_x[t] & 1) * (LBM_TX / 2) + (lx >> 1);
            const int py = (P.tile_y[t] & 1) * (LBM_TY / 2) + (ly >> 1);
            const int ps = pt * LBM_TILE + py * LBM_TX + px, q1 = ls.pp ^ 1;
            C.drho[q1][ps] = 0.25f * a0; C.ux[q1][ps] = a2 / a1; C.uy[q1][ps] = a3 / a1; C.chi[q1][ps] = 0.25f * a4;
        }
    }
}

// ------------------------------------------------------------------ the level kernel
__device__ __forceinline__ bool boundary_cell(const GeneralWork &W)
{
    return (W.fl & (FL_KIND_MASK | FL_SOLID | FL_BNODE)) == (KIND_ACTIVE | FL_BNODE);
}

__device__ __forceinline__ CutLinks cut_links(const RecView &R, const GeneralWork &W, int *status)
{
    CutLinks c;
    const bool b = W.wall && boundary_cell(W);
    const int r = b ? checked_index(W.ax, R.n, status) : 0;
    c.nf = b ? __ldg(R.nfluid + r) : 0u;
#pragma unroll
    for (int q = 0; q < 9; q++) c.v[q] = b ? __ldg(R.v + r * 9 + q) : 0.0f;
    return c;
}

// Shared memory of a block of the level kernel.
template <int KIND, typename T, bool PLAIN> struct LevelShared {
    static constexpr int NW = LBM_BLOCK / 32;
    int nb3[NW][9];                                       // one copy per warp: no block-wide barrier
    WallPair pairs[KIND == 2 ? NW / 2 : 1];
    alignas(16) T pops[PLAIN ? NW : 1][PLAIN ? 9 * 64 : 1];
};

// Warp w of a launch over a level, warp wb of its block.  KIND: 0 no finer level, 1 with a finer
// level, 2 finest level with wall records; ODD: the parity of the in-place population update;
// EDGE: level 0 of a box with edges (or of a mixed batch).
template <int KIND, typename T, bool ODD, bool PLAIN, bool EDGE, bool TIMELINE>
__device__ __forceinline__ void level_warp(const LevelView &P, const LevelView &F, const LevelView &C, const RecView &R,
                                           const StepConsts &k, const LevelStep &ls, LevelShared<KIND, T, PLAIN> &S, int w,
                                           int wb, int lane)
{
    auto wait = [&]() {
        griddep_launch();
        griddep_wait();
        if (TIMELINE) tl_mark(ls.tl, ls.tl_base, 1);
    };
    if (w >= level_warps(P, PLAIN)) return;
    const Lat<T> L{static_cast<T *>(P.f), P.ns, k.pshift};
    if (PLAIN && w >= P.n_gen_warps) {
        const PlainWork W = plain_work(P, ls, w, lane);
        wait();
        plain_warp<T, ODD>(P, C, k, ls, L, W, lane, S.pops[PLAIN ? wb : 0]);
        return;
    }
    const GeneralWork W = general_work(P, C, ls, w, lane, S.nb3[wb]);
    if (KIND == 2 && W.wall && !(wb & 1)) {
        WallPair &wp = S.pairs[KIND == 2 ? wb >> 1 : 0];
        const WallStatic ws = wall_static(R, wp, boundary_cell(W), W.ax, lane, ls.status);
        wait();
        wall_warp(P, R, k, ls, ws, wp, lane);
        pair_arrive(wb >> 1);
        return;
    }
    CutLinks cut;
    if (KIND == 2) cut = cut_links(R, W, ls.status);
    wait();
    general_warp<KIND, T, ODD, PLAIN, EDGE>(P, F, C, R, k, ls, L, W, lane, KIND == 2 && W.wall ? &S.pairs[wb >> 1] : nullptr,
                                     wb >> 1, cut);
}

// Blocks of whole warps (64 or 128 threads, chosen at launch) over the level's work list.
template <int KIND, typename T, bool ODD, bool PLAIN, bool EDGE>
__global__ void __launch_bounds__(LBM_BLOCK, level_min_blocks(KIND, PLAIN, EDGE))
    k_level(LevelView P, LevelView F, LevelView C, RecView R, StepConsts k, LevelStep ls)
{
    __shared__ LevelShared<KIND, T, PLAIN> S;
    const int lane = threadIdx.x & 31, wb = threadIdx.x >> 5;
    tl_mark(ls.tl, ls.tl_base, 0);
    level_warp<KIND, T, ODD, PLAIN, EDGE, true>(P, F, C, R, k, ls, S, blockIdx.x * (blockDim.x >> 5) + wb, wb, lane);
    tl_end(ls.tl, ls.tl_base);
}

// The batched form of k_level: block b belongs to the last solve whose first block is at most b.
__device__ __forceinline__ int batch_member(const BatchArgs &a)
{
    int i = 0;
    for (int m = 1; m < a.n; m++)
        if (a.d[m].first_block <= (int)blockIdx.x) i = m;
    return i;
}

// ... where all members take the same kind of step of the same parity (the serving loop groups by
// level count): the code and the registers of k_level.  With one kernel that selects the kind and
// the parity per block (k_level_batch, all six bodies in it) eight 5-level polar requests took
// 312 us a coarse step, this way 257 (with the prolongations grouped as in a single solve).
template <int KIND, typename T, bool ODD, bool PLAIN, bool EDGE>
__global__ void __launch_bounds__(LBM_BLOCK, level_min_blocks(KIND, PLAIN, EDGE))
    k_level_group(const __grid_constant__ BatchArgs a)
{
    const SolveDesc &d = a.d[batch_member(a)];
    __shared__ LevelShared<KIND, T, PLAIN> S;
    const int lane = threadIdx.x & 31, wb = threadIdx.x >> 5;
    level_warp<KIND, T, ODD, PLAIN, EDGE, false>(d.P, d.F, d.C, d.R, d.k, d.ls, S,
                                                 ((int)blockIdx.x - d.first_block) * (LBM_BLOCK / 32) + wb, wb, lane);
}

// ... and for any mix: the member's kind and parity select the body.
template <typename T>
__global__ void __launch_bounds__(LBM_BLOCK, 5) k_level_batch(const __grid_constant__ BatchArgs a)
{
    const SolveDesc &d = a.d[batch_member(a)];
    __shared__ LevelShared<0, T, false> S0;
    __shared__ LevelShared<1, T, false> S1;
    __shared__ LevelShared<2, T, false> S2;
    const int lane = threadIdx.x & 31, wb = threadIdx.x >> 5, w = ((int)blockIdx.x - d.first_block) * (LBM_BLOCK / 32) + wb;
    const bool odd = d.ls.p != 0;
#define LBM_BATCH_BODY(KIND, ODD) \
    level_warp<KIND, T, ODD, false, true, false>(d.P, d.F, d.C, d.R, d.k, d.ls, S##KIND, w, wb, lane)
    if (d.kind == 2) { if (odd) LBM_BATCH_BODY(2, true); else LBM_BATCH_BODY(2, false); }
    else if (d.kind == 1) { if (odd) LBM_BATCH_BODY(1, true); else LBM_BATCH_BODY(1, false); }
    else { if (odd) LBM_BATCH_BODY(0, true); else LBM_BATCH_BODY(0, false); }
#undef LBM_BATCH_BODY
}

// ------------------------------------------------------------------ launchers
// launch, with programmatic stream serialization when pdl is set (see griddep_wait)
template <typename... Args>
static void launch_pdl_bs(void (*kern)(Args...), unsigned grid, unsigned block, cudaStream_t st, int pdl, Args... args)
{
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(grid);
    cfg.blockDim = dim3(block);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = pdl ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kern, args...);
}

// the level holding the wall records is the finest one, which has no child level
template <typename T, bool ODD, bool PLAIN, bool EDGE>
static void launch_level_e(cudaStream_t st, const LevelView &P, const LevelView &Fv, const LevelView &Cv, bool child,
                           const RecView &R, const StepConsts &k, const LevelStep &ls, const LevelTune &tu)
{
    const int wpb = tu.warps_per_block, warps = level_warps(P, PLAIN);
    const unsigned grid = (unsigned)((warps + wpb - 1) / wpb), bs = 32u * (unsigned)wpb;
    if (ls.wall) launch_pdl_bs(k_level<2, T, ODD, PLAIN, EDGE>, grid, bs, st, tu.pdl, P, Fv, Cv, R, k, ls);
    else if (child) launch_pdl_bs(k_level<1, T, ODD, PLAIN, EDGE>, grid, bs, st, tu.pdl, P, Fv, Cv, R, k, ls);
    else launch_pdl_bs(k_level<0, T, ODD, PLAIN, EDGE>, grid, bs, st, tu.pdl, P, Fv, Cv, R, k, ls);
}

template <typename T, bool ODD>
static void launch_level_t(cudaStream_t st, const LevelView &P, const LevelView &Fv, const LevelView &Cv, bool child,
                           const RecView &R, const StepConsts &k, const LevelStep &ls, const LevelTune &tu)
{
    const bool edge = ls.is_level0 && k.level0_edges;
    if (tu.plain) {
        if (edge) launch_level_e<T, ODD, true, true>(st, P, Fv, Cv, child, R, k, ls, tu);
        else launch_level_e<T, ODD, true, false>(st, P, Fv, Cv, child, R, k, ls, tu);
    } else {
        if (edge) launch_level_e<T, ODD, false, true>(st, P, Fv, Cv, child, R, k, ls, tu);
        else launch_level_e<T, ODD, false, false>(st, P, Fv, Cv, child, R, k, ls, tu);
    }
}

template <typename T>
void launch_level_store(cudaStream_t st, const LevelView &P, const LevelView &Fv, const LevelView &Cv, bool child,
                        const RecView &R, const StepConsts &k, const LevelStep &ls, const LevelTune &tu)
{
    if (ls.p) launch_level_t<T, true>(st, P, Fv, Cv, child, R, k, ls, tu);
    else launch_level_t<T, false>(st, P, Fv, Cv, child, R, k, ls, tu);
}

template <typename T, bool ODD, bool PLAIN, bool EDGE>
static void launch_group_e(cudaStream_t st, const BatchArgs &a, unsigned grid, int pdl)
{
    if (a.kind == 2) launch_pdl_bs(k_level_group<2, T, ODD, PLAIN, EDGE>, grid, LBM_BLOCK, st, pdl, a);
    else if (a.kind == 1) launch_pdl_bs(k_level_group<1, T, ODD, PLAIN, EDGE>, grid, LBM_BLOCK, st, pdl, a);
    else launch_pdl_bs(k_level_group<0, T, ODD, PLAIN, EDGE>, grid, LBM_BLOCK, st, pdl, a);
}

template <typename T, bool ODD> static void launch_group(cudaStream_t st, const BatchArgs &a, unsigned grid, int pdl)
{
    if (a.plain) {
        if (a.edge) launch_group_e<T, ODD, true, true>(st, a, grid, pdl);
        else launch_group_e<T, ODD, true, false>(st, a, grid, pdl);
    } else {
        if (a.edge) launch_group_e<T, ODD, false, true>(st, a, grid, pdl);
        else launch_group_e<T, ODD, false, false>(st, a, grid, pdl);
    }
}

template <typename T> void launch_level_batch_store(cudaStream_t st, const BatchArgs &a, unsigned grid, int pdl)
{
    if (a.kind < 0) launch_pdl_bs(k_level_batch<T>, grid, LBM_BLOCK, st, pdl, a);
    else if (a.odd) launch_group<T, true>(st, a, grid, pdl);
    else launch_group<T, false>(st, a, grid, pdl);
}

}  // namespace lbmdev
