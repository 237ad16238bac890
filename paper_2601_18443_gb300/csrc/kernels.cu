// kernels.cu -- sm_103a kernels around the level step: prolongation, interface transfers of
// set_fields, queries, FP64 reductions, and the launchers of device.cuh.
#include "level.cuh"

namespace lbmdev {

extern template void launch_level_store<float>(cudaStream_t, const LevelView &, const LevelView &, const LevelView &, bool,
                                               const RecView &, const StepConsts &, const LevelStep &, const LevelTune &);
extern template void launch_level_store<__half>(cudaStream_t, const LevelView &, const LevelView &, const LevelView &, bool,
                                                const RecView &, const StepConsts &, const LevelStep &, const LevelTune &);
extern template void launch_level_store<__nv_bfloat16>(cudaStream_t, const LevelView &, const LevelView &, const LevelView &,
                                                       bool, const RecView &, const StepConsts &, const LevelStep &,
                                                       const LevelTune &);
extern template void launch_level_batch_store<float>(cudaStream_t, const BatchArgs &, unsigned, int);
extern template void launch_level_batch_store<__half>(cudaStream_t, const BatchArgs &, unsigned, int);
extern template void launch_level_batch_store<__nv_bfloat16>(cudaStream_t, const BatchArgs &, unsigned, int);

// ------------------------------------------------------------------ prolongation (Sec 2.2)
// ghost children of the band cells of level l: linear LSQ reconstruction of chi and u
// about the parent (fields at time t), rho copied; written to both time levels of l+1.
// One thread a band cell, over the level's list of them: all addresses are static and found
// before the wait for the preceding kernel, so that a launch is one round of loads, the
// arithmetic and the stores (c/256 airfoil, level 4: 1.1 us; 1.8 us with one thread a cell of every
// tile with a band cell, flags and child table read after the wait).  One warp a block spreads the
// scattered accesses over more SMs (blocks of 128: 1.5 us).
#define PROLONG_THREADS 32

struct ProlongCell {
    int s[9];           // own slot and those at offsets +c_q, or s[0] < 0: nothing to do
    int row[2];         // slots of the first child of either row, or -1
};

__device__ __forceinline__ ProlongCell prolong_cell(const LevelView &P, int b)
{
    ProlongCell c;
    c.s[0] = b < P.n_band ? __ldg(P.band_slot + b) : -1;
    c.row[0] = c.row[1] = -1;
    if (c.s[0] < 0) return c;
    c.row[0] = __ldg(P.band_tgt + 4 * b + 1).y;
    c.row[1] = __ldg(P.band_tgt + 4 * b + 2).y;
    const int t = c.s[0] / LBM_TILE, lx = c.s[0] & (LBM_TX - 1), ly = (c.s[0] / LBM_TX) & (LBM_TY - 1);
#pragma unroll
    for (int q = 1; q < 9; q++) {
        const int nx = lx + cxq(q), ny = ly + cyq(q);
        const int sx = nx < 0 ? 0 : (nx >= LBM_TX ? 2 : 1), sy = ny < 0 ? 0 : (ny >= LBM_TY ? 2 : 1);
        const int tt = sx == 1 && sy == 1 ? t : __ldg(P.nbr + t * 9 + dir_of3(sy * 3 + sx));
        c.s[q] = tt < 0 ? c.s[0] : tt * LBM_TILE + (ny & (LBM_TY - 1)) * LBM_TX + (nx & (LBM_TX - 1));
    }
    return c;
}

__device__ __forceinline__ void prolong_write(const LevelView &P, const LevelView &F, int p, const ProlongCell &c)
{
    if (c.s[0] < 0) return;
    Stencil S;
#pragma unroll
    for (int q = 0; q < 9; q++) {
        S.chi[q] = P.chi[p][c.s[q]]; S.ux[q] = P.ux[p][c.s[q]]; S.uy[q] = P.uy[p][c.s[q]];
    }
    const float dr = P.drho[p][c.s[0]];
    float gcx, gcy, gux, guy, gvx, gvy;
    lsq_grad(S.chi, gcx, gcy); lsq_grad(S.ux, gux, guy); lsq_grad(S.uy, gvx, gvy);
#pragma unroll
    for (int b = 0; b < 2; b++) {
        const int cs = c.row[b];
        if (cs < 0) continue;
        float vc[2], vu[2], vv[2];
#pragma unroll
        for (int a = 0; a < 2; a++) {
            const float ox = 0.5f * (a - 0.5f), oy = 0.5f * (b - 0.5f);
            vc[a] = S.chi[0] + gcx * ox + gcy * oy;
            vu[a] = S.ux[0] + gux * ox + guy * oy;
            vv[a] = S.uy[0] + gvx * ox + gvy * oy;
        }
        const float vr[2] = {dr, dr};
#pragma unroll
        for (int h = 0; h < 2; h++) {
            st2(F.chi[h] + cs, vc); st2(F.ux[h] + cs, vu); st2(F.uy[h] + cs, vv); st2(F.drho[h] + cs, vr);
        }
    }
}

__global__ void __launch_bounds__(PROLONG_THREADS) k_prolong(LevelView P, LevelView F, int p, unsigned long long *tl, int tl_base)
{
    tl_mark(tl, tl_base, 0);
    const ProlongCell c = prolong_cell(P, blockIdx.x * PROLONG_THREADS + threadIdx.x);
    griddep_launch();
    griddep_wait();
    tl_mark(tl, tl_base, 1);
    prolong_write(P, F, p, c);
    tl_end(tl, tl_base);
}

// batched form of k_prolong (same solve lookup as k_level_batch)
__global__ void __launch_bounds__(PROLONG_THREADS) k_prolong_batch(const __grid_constant__ ProlongBatchArgs a)
{
    int i = 0;
    for (int m = 1; m < a.n; m++)
        if (a.d[m].first_block <= (int)blockIdx.x) i = m;
    const ProlongDesc &d = a.d[i];
    tl_mark(a.tl, a.tl_base, 0);
    const ProlongCell c = prolong_cell(d.P, ((int)blockIdx.x - d.first_block) * PROLONG_THREADS + threadIdx.x);
    griddep_launch();
    griddep_wait();
    tl_mark(a.tl, a.tl_base, 1);
    prolong_write(d.P, d.F, d.p, c);
    tl_end(a.tl, a.tl_base);
}

// ------------------------------------------------------------------ wall-state query
// The query form of the wall function (one thread a record): it fills the record's state arrays
// and leaves the Newton start of the next step alone, so that queries do not change the
// trajectory.
__global__ void __launch_bounds__(128) k_wallfn(LevelView P, int p, RecView R, StepConsts k)
{
    const int r = blockIdx.x * blockDim.x + threadIdx.x;
    if (r >= R.n) return;
    float drR = 0.f, uR = 0.f, vR = 0.f;
#pragma unroll
    for (int m4 = 0; m4 < 4; m4++)
        wall_gather(P, p, __ldg(reinterpret_cast<const int4 *>(R.st_slot + r * 16) + m4),
                    __ldg(reinterpret_cast<const float4 *>(R.st_wr + r * 16) + m4),
                    __ldg(reinterpret_cast<const float4 *>(R.st_wu + r * 16) + m4), drR, uR, vR, nullptr);
    const WallState w = wall_point(P, R, k, r, R.nx[r], R.ny[r], R.dwb[r], R.utau_start[r], uR, vR);
    R.drhoW[r] = drR; R.uWx[r] = w.uWx; R.uWy[r] = w.uWy; R.utau[r] = w.utau; R.chiB[r] = w.chiB;
    R.tx[r] = w.tx; R.ty[r] = w.ty; R.ut[r] = w.ut;
}

// ------------------------------------------------------------------ interface sync (set_fields)
__global__ void k_restrict(LevelView P, LevelView F, int pp, int pf)
{
    const int t = blockIdx.x, c = threadIdx.x;
    const int slot = t * LBM_TILE + c;
    const uint32_t fl = P.flags[slot];
    if ((fl & FL_KIND_MASK) != KIND_COVERED) return;
    const int cb = child_base(P, t, c & 31, c >> 5);
    if (cb < 0) return;
    float sdr = 0.f, sr = 0.f, sx = 0.f, sy = 0.f, sc = 0.f;
    int n = 0;
    for (int m = 0; m < 4; m++) {
        const int cs = cb + (m & 1) + (m >> 1) * LBM_TX;
        if (F.flags[cs] & FL_SOLID) continue;
        const float dr = F.drho[pf][cs], r = 1.0f + dr;
        sdr += dr; sr += r; sx += r * F.ux[pf][cs]; sy += r * F.uy[pf][cs]; sc += F.chi[pf][cs];
        n++;
    }
    if (n == 0) return;
    P.drho[pp][slot] = sdr / n; P.ux[pp][slot] = sx / sr; P.uy[pp][slot] = sy / sr;
    P.chi[pp][slot] = sc / n;
}

// Logical post-collision populations (f - w, unshifted) of the active fluid cells of a level
// whose next step has parity p, gathered from the in-place layout into out[q * ns + slot]:
// the inverse of put_post.  Values the layout does not keep (populations leaving across the
// inlet or the outlet, or towards a cell without a tile; no step reads them) are NaN.
// Boundary nodes come from their record buffer.  Ghosts report their parent's exploded
// values before an even sub-step and what they relay before an odd one.
template <typename T>
__global__ void k_gather_post(LevelView P, LevelView C, RecView R, StepConsts k, int p, int is_level0, float *out)
{
    __shared__ int nb3[9];
    const int t = blockIdx.x, c = threadIdx.x;
    const int lx = c & 31, ly = c >> 5;
    load_nb3(P, t, nb3);
    __syncthreads();
    const int slot = t * LBM_TILE + c;
    const Lat<T> L{static_cast<T *>(P.f), P.ns, k.pshift};
    const uint32_t fl = P.flags[slot];
    const uint32_t kind = fl & FL_KIND_MASK;
    float o[9];
    for (int q = 0; q < 9; q++) o[q] = NAN;
    if (kind == KIND_GHOST && !(fl & FL_SOLID)) {
        // before an odd sub-step a ghost holds what it relays next (its even sub-step's
        // pulls); before an even one, its parent's exploded values
        const float *eb = C.ebuf + (P.aux[slot] >> 2) * 9;
        for (int q = 0; q < 9; q++) o[q] = p == 1 ? L.ld(oppq(q), slot, q) : eb[q];
    } else if (kind == KIND_ACTIVE && !(fl & FL_SOLID)) {
        if (R.n > 0 && (fl & FL_BNODE) && P.aux) {
            const float *fp = R.fpost + P.aux[slot] * 9;
            for (int q = 0; q < 9; q++) o[q] = fp[q];
        } else if (p == 1) {
            for (int q = 0; q < 9; q++) o[q] = L.ld(oppq(q), slot, q);
        } else {
            int nbs[9];
            const unsigned present = neighbours(nb3, lx, ly, slot, nbs);
            o[0] = L.ld(0, slot, 0);
            const bool edge = is_level0 && k.level0_edges && (fl & (FL_INLET | FL_OUTLET | FL_BOTTOM | FL_TOP));
            const int gi = P.tile_x[t] * LBM_TX + lx, gj = P.tile_y[t] * LBM_TY + ly;
            for (int q = 1; q < 9; q++) {
                if (!edge) {
                    if (present >> q & 1) o[q] = L.ld(q, nbs[q], q);
                } else {
                    const int di = gi + cxq(q), dj = gj + cyq(q);
                    if (di < 0 || di >= k.nx0) continue;
                    if (dj >= 0 && dj < k.ny0) o[q] = L.ld(q, slot0(k, di, dj), q);
                    else o[q] = L.ld(mirror_y(q), slot0(k, di, gj), mirror_y(q));
                }
            }
        }
    }
    for (int q = 0; q < 9; q++) out[(size_t)q * P.ns + slot] = o[q];
}

// Store logical post-collision populations in[q * ns + slot] (f - w) of the active fluid
// cells of a level whose next step has parity p into the in-place layout, the record
// buffers of boundary nodes and the outlet buffer (put_post's writes).  Ghost slots are left
// to the explosion.
template <typename T>
__global__ void k_store_post(LevelView P, RecView R, StepConsts k, int p, int is_level0, const float *in)
{
    __shared__ int nb3[9];
    const int t = blockIdx.x, c = threadIdx.x;
    const int lx = c & 31, ly = c >> 5;
    load_nb3(P, t, nb3);
    __syncthreads();
    const int slot = t * LBM_TILE + c;
    const uint32_t fl = P.flags[slot];
    if ((fl & FL_KIND_MASK) != KIND_ACTIVE || (fl & FL_SOLID)) return;
    const Lat<T> L{static_cast<T *>(P.f), P.ns, k.pshift};
    float o[9];
    for (int q = 0; q < 9; q++) o[q] = in[(size_t)q * P.ns + slot];
    int nbs[9];
    const unsigned present = neighbours(nb3, lx, ly, slot, nbs);
    const bool edge = is_level0 && k.level0_edges && (fl & (FL_INLET | FL_OUTLET | FL_BOTTOM | FL_TOP));
    const int gi = P.tile_x[t] * LBM_TX + lx, gj = P.tile_y[t] * LBM_TY + ly;
    if (p == 0) put_post<T, true>(L, k, slot, nbs, present, edge, gi, gj, o);
    else put_post<T, false>(L, k, slot, nbs, present, edge, gi, gj, o);
    if (R.n > 0 && (fl & FL_BNODE) && P.aux) {
        float *fp = R.fpost + P.aux[slot] * 9;
        for (int q = 0; q < 9; q++) fp[q] = o[q];
    }
    if (is_level0 && k.level0_edges && (fl & (FL_OUTLET | FL_OUTLET2))) put_obuf(k, p, fl, gj, o);
}

// explosion of every band cell of P into the ghosts of F from logical post-collision
// populations post[q * ns + slot] of P
template <typename T>
__global__ void k_explode(LevelView P, LevelView F, StepConsts k, const float *post)
{
    const int t = blockIdx.x, c = threadIdx.x;
    const int slot = t * LBM_TILE + c;
    const uint32_t fl = P.flags[slot];
    if ((fl & FL_KIND_MASK) != KIND_ACTIVE || (fl & FL_SOLID) || !(fl & FL_BAND)) return;
    float o[9];
    for (int q = 0; q < 9; q++) o[q] = post[(size_t)q * P.ns + slot];
    const int b = __ldg(P.aux + slot);
    explode_band<T>(P, F, k, fl, b, band_targets(P, b), o);
}

// rest state: every present cell's populations are e (values to store, relative to the
// storage shift), its fields rho = 1, u = (U, 0), chi = chi_inf
struct Feq9 { float g[9]; };

template <typename T>
__global__ void k_init(LevelView P, Feq9 e, float U, float chi_inf)
{
    const int slot = blockIdx.x * LBM_TILE + threadIdx.x;
    const uint32_t fl = P.flags[slot];
    const bool present = (fl & FL_KIND_MASK) != KIND_ABSENT;
    for (int q = 0; q < 9; q++) PopIO<T>::st(static_cast<T *>(P.f) + (size_t)q * P.ns + slot, present ? e.g[q] : 0.0f);
    for (int h = 0; h < 2; h++) {
        P.drho[h][slot] = 0.0f;
        P.ux[h][slot] = present ? U : 0.0f;
        P.uy[h][slot] = 0.0f;
        P.chi[h][slot] = chi_inf;
    }
}

// n groups of nine values g (side buffers at rest)
__global__ void k_fill9(float *buf, long long n, Feq9 g)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < 9 * n) buf[i] = g.g[i % 9];
}

// ------------------------------------------------------------------ FP64 reductions
__device__ __forceinline__ double warp_sum(double v)
{
    for (int off = 16; off >= 1; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
    return v;
}

// surface loads, eqs 29-30: per segment IDW of C_p and signed C_f from two boundary nodes
__global__ void __launch_bounds__(256) k_loads(LoadsView S, RecView R, float U, double *acc)
{
    __shared__ double red[4][8];
    const int k = blockIdx.x * blockDim.x + threadIdx.x;
    double cfx = 0, cfy = 0, cpx = 0, cpy = 0;
    if (k < S.nseg) {
        const int b1 = S.b1[k], b2 = S.b2[k];
        double cp = 0, cf = 0;
        if (b1 >= 0) {
            const double U2 = (double)U * (double)U;
            const double rho1 = 1.0 + (double)R.drhoW[b1];
            const double cp1 = 2.0 / 3.0 * (double)R.drhoW[b1] / U2;
            const double cf1 = 2.0 * rho1 * (double)R.utau[b1] * (double)R.utau[b1] / U2;
            double w1 = S.w1[k], w2 = 0, cp2 = 0, cf2 = 0;
            if (b2 >= 0) {
                const double rho2 = 1.0 + (double)R.drhoW[b2];
                w2 = S.w2[k];
                cp2 = 2.0 / 3.0 * (double)R.drhoW[b2] / U2;
                cf2 = 2.0 * rho2 * (double)R.utau[b2] * (double)R.utau[b2] / U2;
            }
            cp = (w1 * cp1 + w2 * cp2) / (w1 + w2);
            cf = (w1 * cf1 + w2 * cf2) / (w1 + w2);
            const double sg = ((double)R.tx[b1] * S.tx[k] + (double)R.ty[b1] * S.ty[k]) >= 0.0 ? 1.0 : -1.0;
            cf *= sg;
        }
        S.cp[k] = cp;
        S.cf[k] = cf;
        cfx = cf * S.tx[k] * S.ds[k]; cfy = cf * S.ty[k] * S.ds[k];
        cpx = -cp * S.nx[k] * S.ds[k]; cpy = -cp * S.ny[k] * S.ds[k];
    }
    cfx = warp_sum(cfx); cfy = warp_sum(cfy); cpx = warp_sum(cpx); cpy = warp_sum(cpy);
    const int w = threadIdx.x >> 5, ln = threadIdx.x & 31;
    if (ln == 0) { red[0][w] = cfx; red[1][w] = cfy; red[2][w] = cpx; red[3][w] = cpy; }
    __syncthreads();
    if (threadIdx.x < 4) {
        double s = 0;
        for (int i = 0; i < 8; i++) s += red[threadIdx.x][i];
        atomicAdd(&acc[threadIdx.x], s);
    }
}

__global__ void __launch_bounds__(256) k_mass(LevelView P, int p, double area, double *acc, int *status)
{
    __shared__ double red[8];
    const int slot = blockIdx.x * LBM_TILE + threadIdx.x;
    const uint32_t fl = P.flags[slot];
    double v = 0;
    if ((fl & FL_KIND_MASK) == KIND_ACTIVE && !(fl & FL_SOLID)) {
        const float dr = P.drho[p][slot], u = P.ux[p][slot], w = P.uy[p][slot], x = P.chi[p][slot];
        if (!(isfinite(dr) && isfinite(u) && isfinite(w) && isfinite(x))) atomicOr(status, 1);
        v = area * (1.0 + (double)dr);
    }
    v = warp_sum(v);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        double s = 0;
        for (int i = 0; i < 8; i++) s += red[i];
        atomicAdd(acc, s);
    }
}

// one record of the load history (lbm_set_load_history): the step and eq 30's coefficients
// from the loads' FP64 sums, formed as lbm_get_loads forms them, and the FP64 mass
__global__ void k_hist_push(const double *acc, double *ring, int slot, long long step, double chord)
{
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        double *r = ring + 6 * (size_t)slot;
        const double cdf = acc[0] / chord, cdp = acc[2] / chord;
        r[0] = (double)step;
        r[1] = acc[3] / chord;
        r[2] = cdf + cdp;
        r[3] = cdp;
        r[4] = cdf;
        r[5] = acc[4];
    }
}

void launch_hist_push(cudaStream_t st, const double *acc, double *ring, int slot, long long step, double chord)
{
    k_hist_push<<<1, 32, 0, st>>>(acc, ring, slot, step, chord);
}

// ------------------------------------------------------------------ launchers
void launch_level(cudaStream_t st, const LevelView &P, const LevelView *F, const LevelView *C, const RecView &R,
                  const StepConsts &k, const LevelStep &ls, const LevelTune &tu)
{
    const LevelView Fv = F ? *F : P, Cv = C ? *C : P;
    if (P.n_gen_warps + P.n_plain <= 0) return;
    switch (P.store) {
    case 1: launch_level_store<__half>(st, P, Fv, Cv, F != nullptr, R, k, ls, tu); break;
    case 2: launch_level_store<__nv_bfloat16>(st, P, Fv, Cv, F != nullptr, R, k, ls, tu); break;
    default: launch_level_store<float>(st, P, Fv, Cv, F != nullptr, R, k, ls, tu); break;
    }
}

void launch_level_batch(cudaStream_t st, const BatchArgs &a, int store, unsigned grid, int pdl)
{
    if (grid == 0) return;
    switch (store) {
    case 1: launch_level_batch_store<__half>(st, a, grid, pdl); break;
    case 2: launch_level_batch_store<__nv_bfloat16>(st, a, grid, pdl); break;
    default: launch_level_batch_store<float>(st, a, grid, pdl); break;
    }
}

void launch_prolong_batch(cudaStream_t st, const ProlongBatchArgs &a, unsigned grid, int pdl)
{
    if (grid > 0) launch_pdl_bs(k_prolong_batch, grid, PROLONG_THREADS, st, pdl, a);
}

unsigned prolong_blocks(const LevelView &P) { return (unsigned)((P.n_band + PROLONG_THREADS - 1) / PROLONG_THREADS); }

void launch_prolong(cudaStream_t st, const LevelView &P, const LevelView &F, int p, int pdl, unsigned long long *tl,
                    int tl_base)
{
    const unsigned grid = prolong_blocks(P);
    if (grid > 0) launch_pdl_bs(k_prolong, grid, PROLONG_THREADS, st, pdl, P, F, p, tl, tl_base);
}

void launch_wallfn(cudaStream_t st, const LevelView &P, int p, const RecView &R, const StepConsts &k)
{
    if (R.n <= 0) return;
    k_wallfn<<<(R.n + 127) / 128, 128, 0, st>>>(P, p, R, k);
}

void launch_restrict(cudaStream_t st, const LevelView &P, const LevelView &F, int pp, int pf)
{
    k_restrict<<<P.ntiles, LBM_TILE, 0, st>>>(P, F, pp, pf);
}

template <typename T>
static void launch_aa_util(int what, cudaStream_t st, const LevelView &P, const LevelView &Q, const RecView &R,
                           const StepConsts &k, int p, int is_level0, float *buf)
{
    if (what == 0) k_gather_post<T><<<P.ntiles, LBM_TILE, 0, st>>>(P, Q, R, k, p, is_level0, buf);
    else if (what == 1) k_store_post<T><<<P.ntiles, LBM_TILE, 0, st>>>(P, R, k, p, is_level0, buf);
    else k_explode<T><<<P.ntiles, LBM_TILE, 0, st>>>(P, Q, k, buf);
}

static void launch_aa(int what, cudaStream_t st, const LevelView &P, const LevelView &Q, const RecView &R,
                      const StepConsts &k, int p, int is_level0, float *buf)
{
    if (P.ntiles <= 0) return;
    switch (P.store) {
    case 1: launch_aa_util<__half>(what, st, P, Q, R, k, p, is_level0, buf); break;
    case 2: launch_aa_util<__nv_bfloat16>(what, st, P, Q, R, k, p, is_level0, buf); break;
    default: launch_aa_util<float>(what, st, P, Q, R, k, p, is_level0, buf); break;
    }
}

void launch_gather_post(cudaStream_t st, const LevelView &P, const LevelView *C, const RecView &R, const StepConsts &k,
                        int p, int is_level0, float *out)
{
    launch_aa(0, st, P, C ? *C : P, R, k, p, is_level0, out);
}

void launch_store_post(cudaStream_t st, const LevelView &P, const RecView &R, const StepConsts &k, int p, int is_level0,
                       const float *in)
{
    launch_aa(1, st, P, P, R, k, p, is_level0, const_cast<float *>(in));
}

void launch_explode(cudaStream_t st, const LevelView &P, const LevelView &F, const RecView &R, const StepConsts &k,
                    const float *post)
{
    launch_aa(2, st, P, F, R, k, 0, 0, const_cast<float *>(post));
}

void launch_init_feq(cudaStream_t st, const LevelView &P, const float *feq9, float U, float chi_inf)
{
    Feq9 e;
    for (int q = 0; q < 9; q++) e.g[q] = feq9[q];
    switch (P.store) {
    case 1: k_init<__half><<<P.ntiles, LBM_TILE, 0, st>>>(P, e, U, chi_inf); break;
    case 2: k_init<__nv_bfloat16><<<P.ntiles, LBM_TILE, 0, st>>>(P, e, U, chi_inf); break;
    default: k_init<float><<<P.ntiles, LBM_TILE, 0, st>>>(P, e, U, chi_inf); break;
    }
}

void launch_fill9(cudaStream_t st, float *buf, long long n, const float *g9)
{
    if (n <= 0) return;
    Feq9 e;
    for (int q = 0; q < 9; q++) e.g[q] = g9[q];
    k_fill9<<<(unsigned)((9 * n + 255) / 256), 256, 0, st>>>(buf, n, e);
}

void launch_loads(cudaStream_t st, const LoadsView &S, const RecView &R, float U, double *acc4)
{
    if (S.nseg <= 0) return;
    k_loads<<<(S.nseg + 255) / 256, 256, 0, st>>>(S, R, U, acc4);
}

void launch_mass(cudaStream_t st, const LevelView &P, int p, double area, double *acc, int *status)
{
    k_mass<<<P.ntiles, LBM_TILE, 0, st>>>(P, p, area, acc, status);
}

}  // namespace lbmdev
