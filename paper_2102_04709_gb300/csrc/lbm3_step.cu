// lbm3_step.cu -- sm_103a kernels of one timestep of the three-phase MRT colour-gradient
// lattice Boltzmann model with the characteristic-line wetting condition
// (arXiv:2102.04709, Section II).
//
//   tiles (TX x TY nodes, halo staged in shared memory): fused Eq.(1)-(16): pull-streaming with
//              halfway bounce-back (and the x boundary), densities and phase fields, isotropic
//              gradients (Eq.12), the surface-stress tensor and its divergence (Eq.10), MRT
//              collision with forcing (Eq.1-9, 11), recolouring (Eq.13-15)
//     k_tile     tiles near solids or the domain edge, one per CTA, with the wetting of their
//                solid boundary nodes (Eq.21-22, characteristic lines, FP64 ray geometry)
//     k_step_one, k_step_ring, k_step_tma, k_step_tma16, k_step_plain    pure tiles: no solid
//                within 3 nodes, away from the domain edge
//   k_init     rest-equilibrium initial state written as the pre-image of a pull
//   k_fields   post-streaming densities
//   k_diag     FP64 block partials of mass, centroid, max|u|, min rho, non-finite count
#include <cfloat>
#include <cmath>

#include "lbm3_common.cuh"
#include "lbm3_device.cuh"

namespace lbm3k {

namespace {

// ------------------------------------------------------------------------------------------
// fused step
// ------------------------------------------------------------------------------------------
// Rest populations of unit density as R constants, and the FP64 residuals of the rounded
// constants in the density and energy moments: sum_a fl(w_a) = 1 + kDRho, energy row
// M_1 . fl(w) = -2 + kDE, M_2 . fl(w) = 1 + kDEps (row weights -4 + 3|e|^2 and
// 4 - 21/2 |e|^2 + 9/2 |e|^4).  Moments are taken of f - fl(w), which is exact for
// populations within a factor 2 of fl(w_a) and small otherwise, so that the equilibrium
// deviations e - e_eq and eps - eps_eq carry no O(1) cancellation.
constexpr float kW0 = 4.0f / 9.0f, kW1 = 1.0f / 9.0f, kW5 = 1.0f / 36.0f;
constexpr double kDRho = (double)kW0 + 4.0 * (double)kW1 + 4.0 * (double)kW5 - 1.0;
constexpr double kDE = -4.0 * (double)kW0 - 4.0 * (double)kW1 + 8.0 * (double)kW5 + 2.0;
constexpr double kDEps = 4.0 * (double)kW0 - 8.0 * (double)kW1 + 4.0 * (double)kW5 - 1.0;

// MRT collision with forcing in moment space (the rows of M in Eq.4; M^-1 = M^T diag(1/|row|^2)).
// f: totals f_a; F: interfacial force; returns f_dag in f and the velocity of Eq.(11).  The
// update is applied as f_dag = f + M^-1 dm with dm = -S (m - m_eq) + (I - S/2) M Ftilde, so that
// the rounded constants 1/9, 1/36 ... only scale the small non-equilibrium change (dm_0 = 0).
template <typename R>
__device__ __forceinline__ void collide_mrt(R f[kQ], R rho, R Fx, R Fy, R s1, R& ux, R& uy)
{
    const R d0 = f[0] - kW0;
    const R d1 = f[1] - kW1, d2 = f[2] - kW1, d3 = f[3] - kW1, d4 = f[4] - kW1;
    const R d5 = f[5] - kW5, d6 = f[6] - kW5, d7 = f[7] - kW5, d8 = f[8] - kW5;
    const R b14 = (d1 + d3) + (d2 + d4);
    const R b58 = (d5 + d7) + (d6 + d8);
    const R drho = (d0 + b14) + b58 + (R)kDRho;          // rho - 1
    const R de = (-R(4.0) * d0 - b14 + R(2.0) * b58) + (R)kDE;   // e + 2
    const R deps = (R(4.0) * d0 - R(2.0) * b14 + b58) + (R)kDEps; // eps - 1
    const R jx = (f[1] - f[3]) + (f[5] - f[7]) + (f[8] - f[6]);
    const R qx = -R(2.0) * (f[1] - f[3]) + (f[5] - f[7]) + (f[8] - f[6]);
    const R jy = (f[2] - f[4]) + (f[5] - f[7]) + (f[6] - f[8]);
    const R qy = -R(2.0) * (f[2] - f[4]) + (f[5] - f[7]) + (f[6] - f[8]);
    const R pxx = (f[1] - f[2]) + (f[3] - f[4]);
    const R pxy = (f[5] - f[6]) + (f[7] - f[8]);
    const R irho = __fdividef(R(1.0), rho);  // rounding here only perturbs u by ~1 ulp
    ux = (jx + R(0.5) * Fx) * irho;  // Eq.(11)
    uy = (jy + R(0.5) * Fy) * irho;
    const R u2 = ux * ux + uy * uy;
    const R uF = ux * Fx + uy * Fy;
    // relaxation rates, Eq.(5)-(6) (s1 = 1/tau from the caller)
    const R s4 = __fdividef(R(8.0) * (R(2.0) - s1), R(8.0) - s1);
    const R h1 = R(1.0) - R(0.5) * s1, h4 = R(1.0) - R(0.5) * s4;
    // moment changes: relaxation towards the Eq.(3) equilibrium moments
    // e_eq = rho(-2 + 3u^2), eps_eq = rho(1 - 3u^2), q_eq = -rho u, p_eq = rho(ux^2 - uy^2), rho ux uy,
    // plus the moments of the Eq.(9) forcing vector
    // (0, 6uF, -6uF, Fx, -Fx, Fy, -Fy, 2(uxFx - uyFy), uxFy + uyFx)
    const R dE = -s1 * (de + R(2.0) * drho - R(3.0) * rho * u2) + h1 * R(6.0) * uF;
    const R dEps = -s1 * (deps - drho + R(3.0) * rho * u2) - h1 * R(6.0) * uF;
    const R djx = Fx, djy = Fy;
    const R dqx = -s4 * (qx + rho * ux) - h4 * Fx;
    const R dqy = -s4 * (qy + rho * uy) - h4 * Fy;
    const R dpxx = -s1 * (pxx - rho * (ux * ux - uy * uy)) + h1 * R(2.0) * (ux * Fx - uy * Fy);
    const R dpxy = -s1 * (pxy - rho * ux * uy) + h1 * (ux * Fy + uy * Fx);
    // back to populations
    const R c0 = (R(1.0) / R(9.0)) * (dEps - dE);
    const R ca = -(R(1.0) / R(36.0)) * dE - (R(1.0) / R(18.0)) * dEps;
    const R cd = (R(1.0) / R(18.0)) * dE + (R(1.0) / R(36.0)) * dEps;
    const R X1 = (R(1.0) / R(6.0)) * (djx - dqx), Y1 = (R(1.0) / R(6.0)) * (djy - dqy);
    const R X2 = (R(1.0) / R(6.0)) * djx + (R(1.0) / R(12.0)) * dqx;
    const R Y2 = (R(1.0) / R(6.0)) * djy + (R(1.0) / R(12.0)) * dqy;
    const R P4 = R(0.25) * dpxx, Q4 = R(0.25) * dpxy;
    f[0] += c0;
    f[1] += ca + X1 + P4;
    f[2] += ca + Y1 - P4;
    f[3] += ca - X1 + P4;
    f[4] += ca - Y1 - P4;
    f[5] += cd + X2 + Y2 + Q4;
    f[6] += cd - X2 + Y2 - Q4;
    f[7] += cd - X2 - Y2 + Q4;
    f[8] += cd + X2 - Y2 - Q4;
}

// unit normal of one pair (0 if |G| vanishes)
template <typename R>
__device__ __forceinline__ void pair_normal(R ck, R cl, R gkx, R gky, R glx, R gly, R& nx_, R& ny_)
{
    const R Gx = cl * gkx - ck * glx;
    const R Gy = cl * gky - ck * gly;
    const R G2 = Gx * Gx + Gy * Gy;
    if (G2 > kG2Eps) {
        const R r = rsqrt(G2);
        nx_ = Gx * r;
        ny_ = Gy * r;
    } else {
        nx_ = ny_ = R(0.0);
    }
}

// Eq.(12) derivative weights: d_x psi = (psi_1 - psi_3)/3 + (psi_5 - psi_6 - psi_7 + psi_8)/12
template <int W, typename R>
__device__ __forceinline__ void grad9_df(const float (*h)[W], const float (*l)[W], int cx, int cy,
                                         R& gx, R& gy)
{
    R hx, hy, lx_, ly_;
    {
        const R c1 = h[cy][cx + 1], c3 = h[cy][cx - 1], c2 = h[cy + 1][cx], c4 = h[cy - 1][cx];
        const R c5 = h[cy + 1][cx + 1], c6 = h[cy + 1][cx - 1], c7 = h[cy - 1][cx - 1], c8 = h[cy - 1][cx + 1];
        hx = (R(1.0) / R(3.0)) * (c1 - c3) + (R(1.0) / R(12.0)) * ((c5 - c7) + (c8 - c6));
        hy = (R(1.0) / R(3.0)) * (c2 - c4) + (R(1.0) / R(12.0)) * ((c5 - c7) + (c6 - c8));
    }
    {
        const R c1 = l[cy][cx + 1], c3 = l[cy][cx - 1], c2 = l[cy + 1][cx], c4 = l[cy - 1][cx];
        const R c5 = l[cy + 1][cx + 1], c6 = l[cy + 1][cx - 1], c7 = l[cy - 1][cx - 1], c8 = l[cy - 1][cx + 1];
        lx_ = (R(1.0) / R(3.0)) * (c1 - c3) + (R(1.0) / R(12.0)) * ((c5 - c7) + (c8 - c6));
        ly_ = (R(1.0) / R(3.0)) * (c2 - c4) + (R(1.0) / R(12.0)) * ((c5 - c7) + (c6 - c8));
    }
    gx = hx + lx_;
    gy = hy + ly_;
}

// ---- tensor memory accelerator (bulk tensor copies) and mbarrier, inline PTX ----
__device__ __forceinline__ uint32_t smem_u32(const void* p)
{
    return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count)
{
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init()
{
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void mbar_arrive_expect_tx(uint32_t bar, uint32_t bytes)
{
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint32_t bar, uint32_t parity)
{
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(bar), "r"(parity)
        : "memory");
    return ok != 0;
}
// 3-D tiled load of a box at (x, y, z) into shared memory, completing on the mbarrier; x times
// the element size must be a multiple of 16 bytes
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y, int z,
                                            uint32_t bar)
{
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
        " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
        "l"(map), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}
__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, int x, int y, int z, uint32_t src)
{
    asm volatile("cp.async.bulk.tensor.3d.global.shared::cta.tile.bulk_group [%0, {%1, %2, %3}], [%4];" ::"l"(map),
                 "r"(x), "r"(y), "r"(z), "r"(src)
                 : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
// wait until the committed bulk stores have read their shared-memory source
__device__ __forceinline__ void bulk_wait_read0() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
// make this thread's shared-memory writes visible to the bulk copy engine
__device__ __forceinline__ void fence_proxy_async_smem()
{
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
// polls of an mbarrier before a block gives up draining its bulk copies after a timeout (each
// poll may suspend the thread for a short time; a completed copy takes a few microseconds); the
// first wait for a tile's copies polls Params::wait_polls times (kWaitLimit unless lowered to
// test the timeout path)
constexpr int kWaitLimit = 1 << 22;

// A C_SB node whose wall values are not all within kMixEps of one pure fluid: a fluid-fluid
// interface reaches the wall there (a contact line, or one within a few nodes of it), where the
// lagged wetting feedback amplifies the rounding of single-precision phase fields.  Away from
// such nodes the phase fields near walls are those of one fluid and a float suffices.
constexpr double kMixEps = 1e-6;

// Eq.(12) derivative of a float field held in shared memory
template <int W>
__device__ __forceinline__ void grad9_f(const float (*c)[W], int cx, int cy, float& gx, float& gy)
{
    const float c1 = c[cy][cx + 1], c3 = c[cy][cx - 1], c2 = c[cy + 1][cx], c4 = c[cy - 1][cx];
    const float c5 = c[cy + 1][cx + 1], c6 = c[cy + 1][cx - 1], c7 = c[cy - 1][cx - 1], c8 = c[cy - 1][cx + 1];
    gx = (1.0f / 3.0f) * (c1 - c3) + (1.0f / 12.0f) * ((c5 - c7) + (c8 - c6));
    gy = (1.0f / 3.0f) * (c2 - c4) + (1.0f / 12.0f) * ((c5 - c7) + (c6 - c8));
}

// Block-wide barrier that also reports how many of the three fluids occur in the block's
// phase-field region (present: bit k set where a node holds rho_k != 0).  Where only one fluid
// occurs, the two absent fluids have C_l = 0 exactly at every node, so every pair
// G_kl = C_l grad C_k - C_k grad C_l of Eq.(10) and (13) vanishes: no stress, no force and no
// recolouring term, and skipping the stress phase leaves every bit of the result unchanged.
__device__ __forceinline__ int single_fluid_or(int present)
{
    const int f0 = __syncthreads_or(present & 1);
    const int f1 = __syncthreads_or(present & 2);
    const int f2 = __syncthreads_or(present & 4);
    return (f0 != 0) + (f1 != 0) + (f2 != 0);
}

// The same count with one barrier, for the persistent kernels: each warp ORs its lanes' bits
// into the shared word flags[j & 1] of tile iteration j, the barrier publishes them, and thread 0
// clears the word of the next iteration (nobody writes it before the next tile's barriers).
__device__ __forceinline__ int fluids_present(int present, int* flags, int j, int tid)
{
    const int w = __reduce_or_sync(0xffffffffu, present);
    if ((tid & 31) == 0 && w) atomicOr(&flags[j & 1], w);
    __syncthreads();
    const int v = flags[j & 1];
    if (tid == 0) flags[(j + 1) & 1] = 0;
    return __popc(v & 7);
}

// F_s = div T at (rx, ry) of the stress region: Eq.(10) with the Eq.(12) derivative
template <int RX>
__device__ __forceinline__ void div_stress(const float (*txx)[RX], const float (*txy)[RX],
                                           const float (*tyy)[RX], int rx, int ry, float& Fx, float& Fy)
{
    Fx = (1.0f / 3.0f) * (txx[ry][rx + 1] - txx[ry][rx - 1]) +
         (1.0f / 12.0f) * ((txx[ry + 1][rx + 1] - txx[ry - 1][rx - 1]) + (txx[ry - 1][rx + 1] - txx[ry + 1][rx - 1])) +
         (1.0f / 3.0f) * (txy[ry + 1][rx] - txy[ry - 1][rx]) +
         (1.0f / 12.0f) * ((txy[ry + 1][rx + 1] - txy[ry - 1][rx - 1]) + (txy[ry + 1][rx - 1] - txy[ry - 1][rx + 1]));
    Fy = (1.0f / 3.0f) * (txy[ry][rx + 1] - txy[ry][rx - 1]) +
         (1.0f / 12.0f) * ((txy[ry + 1][rx + 1] - txy[ry - 1][rx - 1]) + (txy[ry - 1][rx + 1] - txy[ry + 1][rx - 1])) +
         (1.0f / 3.0f) * (tyy[ry + 1][rx] - tyy[ry - 1][rx]) +
         (1.0f / 12.0f) * ((tyy[ry + 1][rx + 1] - tyy[ry - 1][rx - 1]) + (tyy[ry + 1][rx - 1] - tyy[ry - 1][rx + 1]));
}

// the recoloured post-collision populations of one node are C_k f_a + w_a (Vx_k e_ax + Vy_k e_ay)
struct Recolour {
    float C[kNF], Vx[kNF], Vy[kNF];
};

// One node: velocity (Eq.11), mixture relaxation (Eq.7), MRT collision with forcing (Eq.1-9)
// applied in place to the 9 post-streaming totals f, and the recolouring coefficients of
// Eq.(13)-(15) from the fluid densities r0..r2 and the colour gradients g = (d C_k / dx, dy).
__device__ __forceinline__ Recolour collide_node(const Params& P, float f[kQ], float r0, float r1, float r2,
                                                 float Fx, float Fy, const float g[6], float& ux, float& uy)
{
    const float rho = (r0 + r1) + r2;
    const float ir = __fdividef(1.0f, rho);
    // fractions as the quotient corrected by its exact FMA residual: a node that holds one fluid
    // gets exactly C = 1, so the recolouring leaves its mass unscaled (r * fl(1/r) can round
    // below 1 every step)
    auto frac = [&](float r) {
        const float q = r * ir;
        return fmaf(fmaf(-q, rho, r), ir, q);
    };
    const float c0 = frac(r0), c1 = frac(r1), c2 = frac(r2);
    float n01x, n01y, n02x, n02y, n12x, n12y;
    pair_normal(c0, c1, g[0], g[1], g[2], g[3], n01x, n01y);
    pair_normal(c0, c2, g[0], g[1], g[4], g[5], n02x, n02y);
    pair_normal(c1, c2, g[2], g[3], g[4], g[5], n12x, n12y);
    // tau = 1/2 + 3 / sum(rho_k / nu_k), so 1/tau = D / (D/2 + 3)
    const float D = (r0 * P.inv_nu0 + r1 * P.inv_nu1) + r2 * P.inv_nu2;
    const float s1 = __fdividef(D, 0.5f * D + 3.0f);
    collide_mrt(f, rho, Fx, Fy, s1, ux, uy);
    const float trip = fminf(35.0f * r0 * r1 * r2 * ir * ir * ir, 1.0f);
    const float b01 = P.beta0 * (1.0f + trip * P.g01) * r0 * r1 * ir;
    const float b02 = P.beta0 * (1.0f + trip * P.g02) * r0 * r2 * ir;
    const float b12 = P.beta0 * (1.0f + trip * P.g12) * r1 * r2 * ir;
    Recolour rc;
    rc.C[0] = c0;
    rc.C[1] = c1;
    rc.C[2] = c2;
    rc.Vx[0] = b01 * n01x + b02 * n02x;
    rc.Vy[0] = b01 * n01y + b02 * n02y;
    rc.Vx[1] = -b01 * n01x + b12 * n12x;
    rc.Vy[1] = -b01 * n01y + b12 * n12y;
    rc.Vx[2] = -b02 * n02x - b12 * n12x;
    rc.Vy[2] = -b02 * n02y - b12 * n12y;
    return rc;
}

// Densities and phase fields of position (cx, cy) of a tile's phase-field region from its 27
// post-streaming populations q; returns which fluids occur there (bit k: rho_k != 0; all three
// for float-float fields, which are never skipped).  df: C_k as hi + lo (TwoSum sums, division
// with its FMA residual), else a float quotient.
template <int CX, int CY>
__device__ __forceinline__ int phase_fields(bool df, const float q[27], float (*ch)[CY][CX], float (*cl)[CY][CX],
                                            float (*rh)[CX], int cx, int cy)
{
    if (df) {
        float rhi[kNF], rlo[kNF];
#pragma unroll
        for (int k = 0; k < kNF; k++) sum9_df(q + 9 * k, rhi[k], rlo[k]);
        float th, tl, sh, sl;
        two_sum(rhi[0], rhi[1], th, tl);
        two_sum(th, rhi[2], sh, sl);
        const float dl = (tl + sl) + ((rlo[0] + rlo[1]) + rlo[2]);
        float dh;
        two_sum(sh, dl, dh, sl);  // rho = dh + sl
#pragma unroll
        for (int k = 0; k < kNF; k++) div_df(rhi[k], rlo[k], dh, sl, ch[k][cy][cx], cl[k][cy][cx]);
        rh[cy][cx] = dh;
        return 7;
    }
    float r[kNF];
#pragma unroll
    for (int k = 0; k < kNF; k++) {
        const float* qk = q + 9 * k;
        r[k] = ((qk[0] + (qk[1] + qk[3])) + (qk[2] + qk[4])) + ((qk[5] + qk[7]) + (qk[6] + qk[8]));
    }
    const float rho = (r[0] + r[1]) + r[2];
    const float ir = __fdividef(1.0f, rho);
#pragma unroll
    for (int k = 0; k < kNF; k++) ch[k][cy][cx] = r[k] * ir;
    rh[cy][cx] = rho;
    return (r[0] != 0.0f ? 1 : 0) | (r[1] != 0.0f ? 2 : 0) | (r[2] != 0.0f ? 4 : 0);
}

// Geometry word of a position of a tile's halo-3 region: the storage index of the node it shows
// (its own, wrapped, or the boundary-column node beyond an open side), the node's class, and
// whether the position lies beyond an open side or an odd number of seams away.
constexpr int kGeoIdx = (1 << 27) - 1;  // 27 nx ny < 2^31
constexpr int kGeoSolid = 1 << 28;      // bit 1 of the class
constexpr int kGeoGhost = 1 << 29;
constexpr int kGeoPar = 1 << 30;
__device__ __forceinline__ int geo_class(int g) { return (g >> 27) & 3; }
__device__ __forceinline__ int geo_word(const Params& P, const uint8_t* __restrict__ type, int X, int Y)
{
    const Loc L = locate(P, X, Y);
    if (L.kind == 1) return kSI << 27;
    return L.idx | (int)(__ldg(type + L.idx) & 3) << 27 | (L.kind == 2 ? kGeoGhost : 0) | (L.par ? kGeoPar : 0);
}

// Eq.(12) gradients (gxk, gyk) and the Eq.(10) stress of position (rx, ry) of the stress region
// of a tile with solids: geometry words t of the halo-3 region, phase fields of the
// phase-field region (halo 2).  At a C_SB centre a neighbour without a value of its own takes
// the extrapolation 2 C(P) - C(P - e_a) (its rounding error carried in the lo word), or C(P)
// when P - e_a has none either; lo words exist only in float-float (df) tiles.
template <int HX, int CX, int CY>
__device__ __forceinline__ void stress_at(const Params& P, const int (*t)[HX], const float (*ch)[CY][CX],
                                          const float (*cl)[CY][CX], const float (*rh)[CX], bool df, int rx,
                                          int ry, float gxk[kNF], float gyk[kNF], float& Txx, float& Txy,
                                          float& Tyy)
{
    const int cx = rx + 1, cy = ry + 1, hx = rx + 2, hy = ry + 2;
    Txx = Txy = Tyy = 0.f;
    const int tc = geo_class(t[hy][hx]);
    if (tc == kSI) {
#pragma unroll
        for (int k = 0; k < kNF; k++) gxk[k] = gyk[k] = 0.0f;
        return;
    }
    const float rho = rh[cy][cx];
    float c[kNF];
#pragma unroll
    for (int k = 0; k < kNF; k++) c[k] = ch[k][cy][cx];
    if (tc == kSB) {
        // where neighbour a takes its value from: itself, or through the centre from the opposite
        // neighbour (bit a of ext), or the centre (bit a of ctr)
        int ext = 0, ctr = 0;
#pragma unroll
        for (int a = 1; a < kQ; a++)
            if (geo_class(t[hy + ey(a)][hx + ex(a)]) == kSI)
                (geo_class(t[hy - ey(a)][hx - ex(a)]) == kSI ? ctr : ext) |= 1 << a;
#pragma unroll 1
        for (int k = 0; k < kNF; k++) {
            float v[kQ], vl[kQ];
            const float h0 = ch[k][cy][cx], l0 = df ? cl[k][cy][cx] : 0.0f;
#pragma unroll
            for (int a = 1; a < kQ; a++) {
                const bool x = ext >> a & 1, c = ctr >> a & 1;
                const int yy = c ? cy : (x ? cy - ey(a) : cy + ey(a)), xx = c ? cx : (x ? cx - ex(a) : cx + ex(a));
                const float oh = ch[k][yy][xx], ol = df ? cl[k][yy][xx] : 0.0f;
                float e;
                two_sum(2.0f * h0, -oh, v[a], e);
                vl[a] = x ? (2.0f * l0 - ol) + e : ol;
                v[a] = x ? v[a] : oh;
            }
            gxk[k] = (1.0f / 3.0f) * (v[1] - v[3]) + (1.0f / 12.0f) * ((v[5] - v[7]) + (v[8] - v[6])) +
                     ((1.0f / 3.0f) * (vl[1] - vl[3]) + (1.0f / 12.0f) * ((vl[5] - vl[7]) + (vl[8] - vl[6])));
            gyk[k] = (1.0f / 3.0f) * (v[2] - v[4]) + (1.0f / 12.0f) * ((v[5] - v[7]) + (v[6] - v[8])) +
                     ((1.0f / 3.0f) * (vl[2] - vl[4]) + (1.0f / 12.0f) * ((vl[5] - vl[7]) + (vl[6] - vl[8])));
        }
    } else if (df) {
#pragma unroll
        for (int k = 0; k < kNF; k++) grad9_df<CX>(ch[k], cl[k], cx, cy, gxk[k], gyk[k]);
    } else {
#pragma unroll
        for (int k = 0; k < kNF; k++) grad9_f<CX>(ch[k], cx, cy, gxk[k], gyk[k]);
    }
    const float rho2 = rho * rho;
    pair_stress(P.sig01, c[0], c[1], gxk[0], gyk[0], gxk[1], gyk[1], rho2, Txx, Txy, Tyy);
    pair_stress(P.sig02, c[0], c[2], gxk[0], gyk[0], gxk[2], gyk[2], rho2, Txx, Txy, Tyy);
    pair_stress(P.sig12, c[1], c[2], gxk[1], gyk[1], gxk[2], gyk[2], rho2, Txx, Txy, Tyy);
}

// ---- what the words of the tiles say (one byte per row of 32 nodes) ----
// Bits 0-2: the fluids that the row's nodes hold; 0 only where it has no fluid node.  Bits 3-4: 0, or
// d + 1 where the row is calm in fluid d: every node's total populations are at least kCalmMin, its
// density at most kCalmRho, and the share C of the two other fluids at most calm_share(), in what is
// stored.  (Bits 5-6 of byte 0: settled_steps.)
//
// Where everything that can reach a node within two links is calm in the same d, the other fluids stay
// traces there: a pulled share is the mean of its sources' with the total populations as weights
// (between 0 and calm_share).  In the FP16 storage the traces' offsets round to 0 and the sources keep
// w_a rho_k: at most 10 times that, 1.4 / (9 / 64).  In BF16 an offset C (f_a - w_a rho) is off by 2^-9 of
// itself: summed over the eight that move, |f_a - w_a rho| is at most f_a + w_a 1.4, so 1 + 10 times the
// pulled total; in the rest population, over a node's own eight, at most 2 x 1.4, 20 times it; 31 x 2^-9 =
// 6 % more.  So a share is at most 2.02e-13 at every fluid node of the phase-field region, and the wall
// values of the C_SB nodes there are compared with 2e-13.  (The pulled total is at least 9 / 64: positive
// and finite.)  A gradient component of such a share is at most three times as large (the extrapolation
// beyond a C_SB node doubles one value and subtracts another), those of C_d are rounding (1e-6) and come
// times a share in G_kl, and |G_kl|^2 <= 18 x (2.02e-13)^2 < 8e-25 for every pair: below kG2Eps, so the
// stress of Eq.(10) and the normals of Eq.(13) are exact zeros.  What the recolouring splits is then C_k f alone, from the node's own
// populations: no halo, no phase fields, no barriers.  Traces spread by a node a step and soon are
// in most tiles (of the 512 x 512 cylinder in 95 % after 1000 steps, of which 5 % hold shares above
// 1e-12): us a step after 1000 steps without and with this, 512 x 512 23.6 / 19.7, the 800 x 375
// pillars 22.8 / 21.2 and after 6000 28.1 / 24.2.
constexpr float kCalmMin = 1.0f / 64.0f, kCalmRho = 1.4f, kCalmWall = 2e-13f;
__host__ __device__ constexpr float calm_share(int store) { return store == kStoreF16 ? 1.9e-14f : 1.9e-13f; }

// the smaller one, or NaN where one is NaN (fminf gives the other number)
__device__ __forceinline__ float min_nan(float a, float b)
{
    float m;
    asm("min.NaN.f32 %0, %1, %2;" : "=f"(m) : "f"(a), "f"(b));
    return m;
}
// a node's part of the above: bits 3-5 the fluids with more than a trace, bit 6 not calm at all; f: the
// total populations that are stored
template <int STORE>
__device__ __forceinline__ int calm_bits(const float f[kQ], float rho, float c0, float c1, float c2)
{
    const float m = min_nan(min_nan(min_nan(min_nan(f[0], f[1]), min_nan(f[2], f[3])),
                                    min_nan(min_nan(f[4], f[5]), min_nan(f[6], f[7]))), f[8]);
    constexpr float T = calm_share(STORE);
    return (fabsf(c0) > T ? 8 : 0) | (fabsf(c1) > T ? 16 : 0) | (fabsf(c2) > T ? 32 : 0) |
           (m >= kCalmMin && rho <= kCalmRho ? 0 : 64);
}
// Whether all populations are numbers.  (A collision keeps their sum, the density: where one of them
// overflows, another is far below 0 or no number.  So a calm node has none that is infinite or NaN.)
__device__ __forceinline__ bool all_finite(const float f[kQ])
{
    bool finite = true;
#pragma unroll
    for (int a = 0; a < kQ; a++) finite = finite && isfinite(f[a]);
    return finite;
}
__device__ __forceinline__ int present_bits(float r0, float r1, float r2)
{
    return (r0 != 0.0f ? 1 : 0) | (r1 != 0.0f ? 2 : 0) | (r2 != 0.0f ? 4 : 0);
}
// The OR of the bits of a row's nodes, by the whole warp (bits 0: no fluid node), with all fluids where a
// collision left infinities or NaN in f: C_k f is NaN there, also for a fluid with C_k = 0.
__device__ __forceinline__ int row_bits(int bits, const float f[kQ])
{
    const int v = __reduce_or_sync(0xffffffffu, bits);
    if (!(v & 64)) return v;
    return __any_sync(0xffffffffu, (bits & 64) && !all_finite(f)) ? v | 7 : v;
}
// the row's byte from that (a row without any density has NaNs in all planes)
__device__ __forceinline__ uint8_t row_byte(int v)
{
    const int d = v >> 3 & 7;
    if (v & 64) return (uint8_t)(v & 7 ? v & 7 : 7);
    return (uint8_t)((v & 7) | (__popc(d) == 1 ? __ffs(d) << 3 : 0));
}

// the fluids that a tile holds
__device__ __forceinline__ int word_fluids(uint64_t b)
{
    b |= b >> 32;
    b |= b >> 16;
    b |= b >> 8;
    return (int)(b & 7u);
}
// d + 1 of the tile's first row with a fluid node (0: not calm)
__device__ __forceinline__ int word_calm(uint64_t b)
{
    const uint64_t rows = (b | b >> 1 | b >> 2) & 0x0101010101010101ull;
    return rows ? (int)(b >> (__ffsll((long long)rows) + 2) & 3u) : 0;
}
// whether every row with a fluid node is calm in fluid d1 - 1
__device__ __forceinline__ bool word_calm_in(uint64_t b, int d1)
{
    const uint64_t rows = (b | b >> 1 | b >> 2) & 0x0101010101010101ull;
    return d1 > 0 && !((b ^ 0x0808080808080808ull * (uint64_t)d1) & (rows << 3 | rows << 4));
}

// How a tile that lies inside the domain can be done, from the words of the 3 x 3 tiles around it:
// the fluids stored there (bits 0-2), and bit 3 where all is calm in one fluid.
__device__ __forceinline__ int fluids_around(const uint64_t* __restrict__ pres, int tile, int ntx)
{
    const int d1 = word_calm(pres[tile]);
    uint64_t nb = 0;
    bool calm = true;
#pragma unroll
    for (int m = 0; m < 9; m++) {
        const uint64_t b = pres[tile + (m / 3 - 1) * ntx + m % 3 - 1];
        nb |= b;
        calm = calm && word_calm_in(b, d1);
    }
    return word_fluids(nb) | (calm ? 8 : 0);
}
// the same, by a whole warp with one word per lane
__device__ __forceinline__ int fluids_around_warp(const uint64_t* __restrict__ pres, int tile, int ntx, int lane)
{
    uint64_t b = 0;
    if (lane < 9) b = pres[tile + (lane / 3 - 1) * ntx + lane % 3 - 1];
    const int d1 = __shfl_sync(0xffffffffu, word_calm(b), 4);
    const bool calm = __all_sync(0xffffffffu, lane >= 9 || word_calm_in(b, d1));
    return __reduce_or_sync(0xffffffffu, word_fluids(b)) | (calm ? 8 : 0);
}
// one fluid: k_step_one's tiles
__device__ __forceinline__ bool one_fluid(int around) { return __popc((unsigned)around & 7u) == 1; }
__global__ void k_count(const Params P, const int* __restrict__ tiles, const int ntiles,
                        const uint64_t* __restrict__ pres, unsigned* __restrict__ out)
{
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    const bool several = t < ntiles && !one_fluid(fluids_around(pres, tiles[t], (P.nx + kTX - 1) / kTX));
    const unsigned n = __popc(__ballot_sync(0xffffffffu, several));
    if ((threadIdx.x & 31) == 0 && n) atomicAdd(out, n);
}
// In the list of tiles of the kernels that move all 27 planes: the tile is calm, no gradients needed.
constexpr int kCalmTile = 1 << 30;

// Eq.(10) stress on the halo-1 region of a pure tile from the phase fields of its halo-2 region
// (float path: no solid, no float-float words)
template <int TX, int TY>
__device__ __forceinline__ void stress_halo1(const Params& P, const float (*s_ch)[TY + 4][TX + 4],
                                             const float (*s_rho)[TX + 4], float (*s_txx)[TX + 2],
                                             float (*s_txy)[TX + 2], float (*s_tyy)[TX + 2], int tid)
{
    constexpr int CX = TX + 4, RX = TX + 2, RY = TY + 2;
    for (int r = tid; r < RX * RY; r += TX * TY) {
        const int rx = r % RX, ry = r / RX;
        const int cx = rx + 1, cy = ry + 1;
        const float rho = s_rho[cy][cx];
        float c[kNF], gxk[kNF], gyk[kNF];
#pragma unroll
        for (int k = 0; k < kNF; k++) {
            c[k] = s_ch[k][cy][cx];
            grad9_f<CX>(s_ch[k], cx, cy, gxk[k], gyk[k]);
        }
        float Txx = 0.f, Txy = 0.f, Tyy = 0.f;
        const float rho2 = rho * rho;
        pair_stress(P.sig01, c[0], c[1], gxk[0], gyk[0], gxk[1], gyk[1], rho2, Txx, Txy, Tyy);
        pair_stress(P.sig02, c[0], c[2], gxk[0], gyk[0], gxk[2], gyk[2], rho2, Txx, Txy, Tyy);
        pair_stress(P.sig12, c[1], c[2], gxk[1], gyk[1], gxk[2], gyk[2], rho2, Txx, Txy, Tyy);
        s_txx[ry][rx] = Txx;
        s_txy[ry][rx] = Txy;
        s_tyy[ry][rx] = Tyy;
    }
}

// Pure FP32 tiles through the tensor memory accelerator, persistent: block b handles tiles
// b, b + gridDim.x, ...  For each tile the 27 pull-source planes over the (TX + 8) x (TY + 6)
// box starting at (x0 - 4, y0 - 3) -- x rounded down to a 16-byte boundary -- arrive by one bulk
// tensor copy completing on an mbarrier, and the pulls read them at compile-time offsets.  The
// box is needed only for the pulls: as soon as they are done the copy of the next tile's box is
// issued, so it lands while this tile computes its stress, force, collision and recolouring.
// The 27 output planes are written directly (STAGE = false: 72 KB of shared memory per block)
// or staged in shared memory and written by one bulk tensor store per tile (STAGE = true,
// 100 KB).  kTmaBlocksPerSm = 2 blocks per SM: three (the most that fit) measured slower.
// pres_out gets "all fluids" for its tiles: it looks at no words, but the launches that take over
// when the copy-wait limit is changed do.
// Same arithmetic as k_step_plain, so the two give identical results.
template <int TX, int TY, bool STAGE>
__global__ void __launch_bounds__(TX* TY, kTmaBlocksPerSm) k_step_tma(const Params P, const int* __restrict__ tiles,
                                                        const int ntiles, float* __restrict__ fout,
                                                        float* __restrict__ uout,
                                                        const __grid_constant__ CUtensorMap tm_in_a,
                                                        const __grid_constant__ CUtensorMap tm_in_b,
                                                        const __grid_constant__ CUtensorMap tm_out,
                                                        uint64_t* __restrict__ pres_out)
{
    constexpr int NT = TX * TY;
    constexpr int CX = TX + 4, CY = TY + 4;  // phase-field region (halo 2)
    constexpr int RX = TX + 2, RY = TY + 2;  // stress region (halo 1)
    constexpr int BX = TX + 8, BY = TY + 6;  // pull-source box
    constexpr int NBOX = kQ * kNF * BY * BX;
    constexpr int NBOXP = (NBOX + 31) / 32 * 32;  // keeps the staging buffer 128-byte aligned
    constexpr int NRING = CX * CY - TX * TY;      // halo-2 ring: one node per thread at most
    static_assert(NRING <= NT, "the ring of the halo-2 region must not exceed one node per thread");
    static_assert((kTmaPlanesA * BY * BX * 4) % 128 == 0, "second copy must start 128-byte aligned");
    __shared__ float s_ch[kNF][CY][CX];
    __shared__ float s_rho[CY][CX];
    __shared__ float s_txx[RY][RX], s_txy[RY][RX], s_tyy[RY][RX];
    __shared__ __align__(8) uint64_t s_bar[2];  // completion of copy A (planes 0..13) and B (14..26)
    __shared__ int s_flags[2];                  // fluids present in the tile, by iteration parity
    extern __shared__ unsigned char dsm[];
    float* box = reinterpret_cast<float*>(dsm + ((128u - (smem_u32(dsm) & 127u)) & 127u));  // [27][BY][BX]
    float* outb = box + NBOXP;                                                              // [27][TY][TX]

    const int tid = threadIdx.x + TX * threadIdx.y;
    const int lx = threadIdx.x, ly = threadIdx.y;
    const int ntx = (P.nx + TX - 1) / TX;
    const uint32_t bar_a = smem_u32(&s_bar[0]), bar_b = smem_u32(&s_bar[1]);
    if ((int)blockIdx.x >= ntiles) return;
    auto issue_a = [&](int tile) {
        const int x0 = (tile % ntx) * TX, y0 = (tile / ntx) * TY;
        mbar_arrive_expect_tx(bar_a, (uint32_t)(kTmaPlanesA * BY * BX) * 4u);
        tma_load_3d(smem_u32(box), &tm_in_a, x0 - 4, y0 - 3, 0, bar_a);
    };
    auto issue_b = [&](int tile) {
        const int x0 = (tile % ntx) * TX, y0 = (tile / ntx) * TY;
        mbar_arrive_expect_tx(bar_b, (uint32_t)((kQ * kNF - kTmaPlanesA) * BY * BX) * 4u);
        tma_load_3d(smem_u32(box + kTmaPlanesA * BY * BX), &tm_in_b, x0 - 4, y0 - 3, kTmaPlanesA, bar_b);
    };
    int tile = tiles[blockIdx.x];
    int last_a = 0, last_b = 0;  // tile iteration of the latest copy into each part (thread 0)
    if (tid == 0) {
        mbar_init(bar_a, 1);
        mbar_init(bar_b, 1);
        fence_mbar_init();
        issue_a(tile);
        issue_b(tile);
        s_flags[0] = s_flags[1] = 0;
    }
    __syncthreads();

    // bounded wait for one part of iteration j's box, with the same outcome in every thread; on
    // a timeout the error bit is set and thread 0 gives the copies it issued a second bounded
    // wait, so that none lands in a later block's shared memory
    auto wait_part = [&](uint32_t bar, int j) -> bool {
        bool ok = false;
        for (int it = 0; it < P.wait_polls && !ok; it++) ok = mbar_try_wait(bar, j & 1);
        if (!__syncthreads_or(!ok)) return true;
        if (tid == 0) {
            atomicOr(P.err, 1);
            for (int it = 0; it < kWaitLimit && !mbar_try_wait(bar_a, last_a & 1); it++) {
            }
            for (int it = 0; it < kWaitLimit && !mbar_try_wait(bar_b, last_b & 1); it++) {
            }
            bulk_wait_read0();
        }
        return false;
    };
    // pulls of the node at (cx, cy) of the phase-field region from the planes p of the box with
    // P0 <= p < P1 (q[p], p = 9 k + a)
    auto pull = [&](int cx, int cy, float q[27], int p0, int p1) {
#pragma unroll
        for (int p = 0; p < kQ * kNF; p++) {
            const int a = p % kQ;
            if (p >= p0 && p < p1) q[p] = box[(p * BY + cy + 1 - ey(a)) * BX + cx + 2 - ex(a)];
        }
    };
    // densities and phase fields of one node; returns which fluids it holds (bit k: rho_k != 0)
    auto store_phase = [&](int cx, int cy, float r0, float r1, float r2) {
        const float rho = (r0 + r1) + r2;
        const float ir = __fdividef(1.0f, rho);
        s_ch[0][cy][cx] = r0 * ir;
        s_ch[1][cy][cx] = r1 * ir;
        s_ch[2][cy][cx] = r2 * ir;
        s_rho[cy][cx] = rho;
        return (r0 != 0.0f ? 1 : 0) | (r1 != 0.0f ? 2 : 0) | (r2 != 0.0f ? 4 : 0);
    };

    // the ring node of this thread (a fixed position in every tile)
    const bool ring = tid < NRING;
    int rcx = 0, rcy = 0;
    if (ring) {
        if (tid < 2 * CX) {
            rcx = tid % CX;
            rcy = tid / CX;
        } else if (tid < 4 * CX) {
            rcx = (tid - 2 * CX) % CX;
            rcy = CY - 2 + (tid - 2 * CX) / CX;
        } else {
            const int rr0 = tid - 4 * CX;  // 4 * TY side nodes
            const int side = rr0 / (2 * TY), rr = rr0 % (2 * TY);
            rcy = 2 + rr / 2;
            rcx = side == 0 ? (rr & 1) : CX - 2 + (rr & 1);
        }
    }

    int j = 0;
    for (int t = blockIdx.x; t < ntiles; t += gridDim.x, j++) {
        // the next tile's index is read now and used after the pulls
        const bool more = t + (int)gridDim.x < ntiles;
        const int next = more ? tiles[t + gridDim.x] : 0;
        const int x0 = (tile % ntx) * TX, y0 = (tile / ntx) * TY;

        // ---- phase 1: pulls, densities and phase fields of the halo-2 region, in two passes
        // over the two parts of the box (the sums keep the order of the one-pass kernel) ----
        if (!wait_part(bar_a, j)) return;
        float q[27];
        float ra0 = 0.0f, ra1 = 0.0f;  // ring node: rho_0 and the planes 9..13 part of rho_1
        if (ring) {
            pull(rcx, rcy, q, 0, kTmaPlanesA);
            ra0 = ((q[0] + (q[1] + q[3])) + (q[2] + q[4])) + ((q[5] + q[7]) + (q[6] + q[8]));
            ra1 = (q[9] + (q[10] + q[12])) + (q[11] + q[13]);
        }
        float f[kQ], r0, r1, r2;
        pull(lx + 2, ly + 2, q, 0, kTmaPlanesA);
#pragma unroll
        for (int a = 0; a < kQ; a++) f[a] = a < 5 ? q[a] + q[9 + a] : q[a];
        r0 = ((q[0] + (q[1] + q[3])) + (q[2] + q[4])) + ((q[5] + q[7]) + (q[6] + q[8]));
        r1 = (q[9] + (q[10] + q[12])) + (q[11] + q[13]);
        // the wait for part B is a barrier: past it every thread has pulled from part A, which
        // is then free for the next tile's copy while part B is pulled and this tile computes
        if (!wait_part(bar_b, j)) return;
        if (tid == 0 && more) {
            issue_a(next);
            last_a = j + 1;
        }
        int present = 0;
        if (ring) {
            pull(rcx, rcy, q, kTmaPlanesA, kQ * kNF);
            const float rb1 = ra1 + ((q[14] + q[16]) + (q[15] + q[17]));
            const float rb2 = ((q[18] + (q[19] + q[21])) + (q[20] + q[22])) + ((q[23] + q[25]) + (q[24] + q[26]));
            present |= store_phase(rcx, rcy, ra0, rb1, rb2);
        }
        pull(lx + 2, ly + 2, q, kTmaPlanesA, kQ * kNF);
#pragma unroll
        for (int a = 0; a < kQ; a++) f[a] = (a < 5 ? f[a] : f[a] + q[9 + a]) + q[18 + a];
        r1 = r1 + ((q[14] + q[16]) + (q[15] + q[17]));
        r2 = ((q[18] + (q[19] + q[21])) + (q[20] + q[22])) + ((q[23] + q[25]) + (q[24] + q[26]));
        present |= store_phase(lx + 2, ly + 2, r0, r1, r2);
        const bool mixed = fluids_present(present, s_flags, j, tid) != 1;
        if (tid == 0 && more) {
            issue_b(next);
            last_b = j + 1;
        }

        // ---- phase 2: stress tensor of Eq.(10) on the halo-1 region ----
        if (mixed) stress_halo1<TX, TY>(P, s_ch, s_rho, s_txx, s_txy, s_tyy, tid);
        // the previous tile's bulk store must have read the staging buffer before it is refilled
        if (STAGE && tid == 0) bulk_wait_read0();
        __syncthreads();

        // ---- phase 3: force, collision, recolouring into the staging buffer ----
        float Fx = 0.0f, Fy = 0.0f, g[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
        if (mixed) {
            div_stress<RX>(s_txx, s_txy, s_tyy, lx + 1, ly + 1, Fx, Fy);
            // own colour gradients, the same stencil as phase 2 on the same phase fields (the
            // next tile overwrites them only after the barrier at the top of the loop)
#pragma unroll
            for (int k = 0; k < kNF; k++) grad9_f<CX>(s_ch[k], lx + 2, ly + 2, g[2 * k], g[2 * k + 1]);
        }
        float ux, uy;
        const Recolour rc = collide_node(P, f, r0, r1, r2, Fx, Fy, g, ux, uy);
        if (uout) {
            const int i = (y0 + ly) * P.nx + x0 + lx;
            uout[i] = ux;
            uout[P.N + i] = uy;
        }
        // (what the tile's rows hold is not looked at: all fluids, and not calm)
        if (tid == 0) pres_out[tile] = 0x0707070707070707ull;
        tile = next;
        if constexpr (STAGE) {
            float* o = outb + ly * TX + lx;
#pragma unroll
            for (int k = 0; k < kNF; k++)
#pragma unroll
                for (int a = 0; a < kQ; a++)
                    o[(k * kQ + a) * TY * TX] =
                        rc.C[k] * f[a] + wq(a) * (rc.Vx[k] * (float)ex(a) + rc.Vy[k] * (float)ey(a));
            fence_proxy_async_smem();
            __syncthreads();
            if (tid == 0) {
                tma_store_3d(&tm_out, x0, y0, 0, smem_u32(outb));
                bulk_commit();
            }
        } else {
            float* o = fout + (y0 + ly) * P.nx + x0 + lx;
#pragma unroll
            for (int k = 0; k < kNF; k++)
#pragma unroll
                for (int a = 0; a < kQ; a++)
                    o[P.off_plane[k * kQ + a]] =
                        rc.C[k] * f[a] + wq(a) * (rc.Vx[k] * (float)ex(a) + rc.Vy[k] * (float)ey(a));
        }
    }
    if (STAGE && tid == 0) bulk_wait_read0();
}

// ---- named barriers of one consumer group and a plain mbarrier arrival ----
__device__ __forceinline__ void group_sync(int id, int nthreads)
{
    asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(nthreads) : "memory");
}
// barrier of the group that also ORs a predicate over its threads
__device__ __forceinline__ bool group_or(bool v, int id, int nthreads)
{
    uint32_t r;
    asm volatile(
        "{\n\t.reg .pred p, q;\n\t"
        "setp.ne.u32 p, %1, 0;\n\t"
        "bar.red.or.pred q, %2, %3, p;\n\t"
        "selp.u32 %0, 1, 0, q;\n\t}"
        : "=r"(r)
        : "r"((uint32_t)v), "r"(id), "r"(nthreads)
        : "memory");
    return r != 0;
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar)
{
    asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(bar) : "memory");
}

// collide_mrt without a force, for nodes that hold one fluid: the terms of F are exact zeros there,
// so leaving them out changes no bit of the result (but for the sign of a zero).  __fmul_rn where
// the product is rounded there before the (zero) term is added, so that it is not fused here.
__device__ __forceinline__ void collide_mrt_free(float f[kQ], float rho, float s1, float& ux, float& uy)
{
    const float d0 = f[0] - kW0;
    const float d1 = f[1] - kW1, d2 = f[2] - kW1, d3 = f[3] - kW1, d4 = f[4] - kW1;
    const float d5 = f[5] - kW5, d6 = f[6] - kW5, d7 = f[7] - kW5, d8 = f[8] - kW5;
    const float b14 = (d1 + d3) + (d2 + d4);
    const float b58 = (d5 + d7) + (d6 + d8);
    const float drho = (d0 + b14) + b58 + (float)kDRho;
    const float de = (-4.0f * d0 - b14 + 2.0f * b58) + (float)kDE;
    const float deps = (4.0f * d0 - 2.0f * b14 + b58) + (float)kDEps;
    const float jx = (f[1] - f[3]) + (f[5] - f[7]) + (f[8] - f[6]);
    const float qx = -2.0f * (f[1] - f[3]) + (f[5] - f[7]) + (f[8] - f[6]);
    const float jy = (f[2] - f[4]) + (f[5] - f[7]) + (f[6] - f[8]);
    const float qy = -2.0f * (f[2] - f[4]) + (f[5] - f[7]) + (f[6] - f[8]);
    const float pxx = (f[1] - f[2]) + (f[3] - f[4]);
    const float pxy = (f[5] - f[6]) + (f[7] - f[8]);
    const float irho = __fdividef(1.0f, rho);
    ux = __fmul_rn(jx, irho);
    uy = __fmul_rn(jy, irho);
    const float u2 = ux * ux + uy * uy;
    const float s4 = __fdividef(8.0f * (2.0f - s1), 8.0f - s1);
    const float dE = __fmul_rn(-s1, de + 2.0f * drho - 3.0f * rho * u2);
    const float dEps = __fmul_rn(-s1, deps - drho + 3.0f * rho * u2);
    const float dqx = __fmul_rn(-s4, qx + rho * ux);
    const float dqy = __fmul_rn(-s4, qy + rho * uy);
    const float dpxx = __fmul_rn(-s1, pxx - rho * (ux * ux - uy * uy));
    const float dpxy = __fmul_rn(-s1, pxy - rho * ux * uy);
    const float c0 = (1.0f / 9.0f) * (dEps - dE);
    const float ca = -(1.0f / 36.0f) * dE - (1.0f / 18.0f) * dEps;
    const float cd = (1.0f / 18.0f) * dE + (1.0f / 36.0f) * dEps;
    const float X1 = (1.0f / 6.0f) * -dqx, Y1 = (1.0f / 6.0f) * -dqy;
    const float X2 = __fmul_rn(1.0f / 12.0f, dqx), Y2 = __fmul_rn(1.0f / 12.0f, dqy);
    const float P4 = 0.25f * dpxx, Q4 = 0.25f * dpxy;
    f[0] += c0;
    f[1] += ca + X1 + P4;
    f[2] += ca + Y1 - P4;
    f[3] += ca - X1 + P4;
    f[4] += ca - Y1 - P4;
    f[5] += cd + X2 + Y2 + Q4;
    f[6] += cd - X2 + Y2 - Q4;
    f[7] += cd - X2 - Y2 + Q4;
    f[8] += cd + X2 - Y2 - Q4;
}

// fraction r / rho of a fluid as collide_node forms it: the quotient corrected by its FMA residual
__device__ __forceinline__ float fraction(float r, float rho)
{
    const float ir = __fdividef(1.0f, rho);
    const float q = r * ir;
    return fmaf(fmaf(-q, rho, r), ir, q);
}

// density of one fluid from its 9 post-streaming populations, in the order of phase_fields
__device__ __forceinline__ float sum9(const float* q)
{
    return ((q[0] + (q[1] + q[3])) + (q[2] + q[4])) + ((q[5] + q[7]) + (q[6] + q[8]));
}

// write c f_a as the populations of fluid l of node i
template <int STORE>
__device__ __forceinline__ void store_fluid(const Params& P, const Pop& out, int l, int i, const float f[kQ], float c)
{
    const int N = (int)P.N;
    if constexpr (STORE == kStoreF32) {
        float* o = out.f + i + l * kQ * N;
#pragma unroll
        for (int a = 0; a < kQ; a++) o[P.off_plane[a]] = c * f[a];
    } else {
        float v[kQ];
#pragma unroll
        for (int a = 0; a < kQ; a++) v[a] = __fmul_rn(c, f[a]);  // rounded here, as store_node gets it
        const float r = ((v[0] + (v[1] + v[3])) + (v[2] + v[4])) + ((v[5] + v[7]) + (v[6] + v[8]));
        out.rho[l * N + i] = r;
#pragma unroll
        for (int a = 1; a < kQ; a++) out.off[(8 * l + a - 1) * N + i] = enc16<STORE>(v[a] - wq(a) * r);
    }
}

// One node that holds fluid k alone, from the 9 post-streaming populations f of that fluid: its
// velocity and, in f, its post-collision populations; the same bits as collide_node and the
// recolouring give with the other two fluids' zeros.  false where they would not be, as it spreads to
// the populations of the absent fluids too: a density whose fraction does not come out as 1 (a zero, an
// infinity or a NaN).  So does what all_single looks for.
__device__ __forceinline__ bool collide_single(const Params& P, int k, float f[kQ], float r, float& ux, float& uy)
{
    const float c = fraction(r, r);
    const float D = r * (k == 0 ? P.inv_nu0 : (k == 1 ? P.inv_nu1 : P.inv_nu2));
    const float s1 = __fdividef(D, 0.5f * D + 3.0f);
    collide_mrt_free(f, r, s1, ux, uy);
    return c == 1.0f;
}
// Whether that holds at every node of a row, by the whole warp: plain (what collide_single says), and no
// infinity or NaN among the populations f after the collision.  still: whether the node is calm, then whether
// all are; only where they are not is f looked at.  Nodes that take no part: both true.
__device__ __forceinline__ bool all_single(bool plain, bool& still, const float f[kQ])
{
    const bool mine = still;
    still = __all_sync(0xffffffffu, still);
    if (!still) plain = plain && (mine || all_finite(f));
    return __all_sync(0xffffffffu, plain);
}

// One node at which |G_kl| vanishes for every pair (see calm_bits), from its 9 post-streaming totals f
// and densities: collide_node without force and normals, and the recolouring, to the planes of the
// fluids in write.  Returns its bits for row_byte.
template <int STORE>
__device__ __forceinline__ int collide_calm(const Params& P, const Pop& fout, float* uout, int i, float f[kQ], float r0,
                                            float r1, float r2, int write)
{
    const float rho = (r0 + r1) + r2;
    const float c[kNF] = {fraction(r0, rho), fraction(r1, rho), fraction(r2, rho)};
    const float D = (r0 * P.inv_nu0 + r1 * P.inv_nu1) + r2 * P.inv_nu2;
    const float s1 = __fdividef(D, 0.5f * D + 3.0f);
    float ux, uy;
    collide_mrt_free(f, rho, s1, ux, uy);
    if (uout) {
        uout[i] = ux;
        uout[P.N + i] = uy;
    }
#pragma unroll
    for (int l = 0; l < kNF; l++)
        if (write >> l & 1) store_fluid<STORE>(P, fout, l, i, f, c[l]);
    return present_bits(r0, r1, r2) | calm_bits<STORE>(f, rho, c[0], c[1], c[2]);
}

// the bits of a recoloured node for row_byte (one that the recolouring shifts is not calm: its traces are
// not C_k f)
template <int STORE>
__device__ __forceinline__ int recoloured_bits(const float f[kQ], float r0, float r1, float r2, const Recolour& rc)
{
    const bool shifts = rc.Vx[0] != 0.0f || rc.Vy[0] != 0.0f || rc.Vx[1] != 0.0f || rc.Vy[1] != 0.0f ||
                        rc.Vx[2] != 0.0f || rc.Vy[2] != 0.0f;
    return present_bits(r0, r1, r2) | calm_bits<STORE>(f, (r0 + r1) + r2, rc.C[0], rc.C[1], rc.C[2]) | (shifts ? 64 : 0);
}

// write the 27 recoloured post-collision populations of node i
template <int STORE>
__device__ __forceinline__ void store_recoloured(const Params& P, const Pop& out, int i, const float f[kQ],
                                                 const Recolour& rc)
{
    if constexpr (STORE == kStoreF32) {
        float* o = out.f + i;
#pragma unroll
        for (int k = 0; k < kNF; k++)
#pragma unroll
            for (int a = 0; a < kQ; a++)
                o[P.off_plane[k * kQ + a]] =
                    rc.C[k] * f[a] + wq(a) * (rc.Vx[k] * (float)ex(a) + rc.Vy[k] * (float)ey(a));
    } else {
        float v[27];
#pragma unroll
        for (int k = 0; k < kNF; k++)
#pragma unroll
            for (int a = 0; a < kQ; a++)
                v[9 * k + a] = rc.C[k] * f[a] + wq(a) * (rc.Vx[k] * (float)ex(a) + rc.Vy[k] * (float)ey(a));
        store_node<STORE>(out, P.N, i, v);
    }
}

// position j of the ring that the halo-2 region of a tile has around the tile's own nodes
template <int TX, int TY>
__device__ __forceinline__ void ring_position(int j, int& cx, int& cy)
{
    constexpr int CX = TX + 4, CY = TY + 4;
    if (j < 2 * CX) {
        cx = j % CX;
        cy = j / CX;
    } else if (j < 4 * CX) {
        cx = (j - 2 * CX) % CX;
        cy = CY - 2 + (j - 2 * CX) / CX;
    } else {
        const int r = j - 4 * CX;  // 4 * TY side nodes
        const int side = r / (2 * TY), rr = r % (2 * TY);
        cy = 2 + rr / 2;
        cx = side == 0 ? (rr & 1) : CX - 2 + (rr & 1);
    }
}

// Pure tiles by plain loads (nx not a multiple of what the bulk copies need): one CTA per TX x TY
// tile.  Pull-streaming of every node of the halo-2 region (densities and phase fields C_k; the
// tile's own nodes keep their 9 post-streaming totals and 3 densities in registers), the Eq.(10)
// stress on the halo-1 region, then force, velocity, MRT collision with forcing, recolouring and 27
// stores per node.  all: take the tiles with one fluid around too, which are k_step_one's otherwise.
template <int TX, int TY, int STORE>
__global__ void __launch_bounds__(TX* TY, 4) k_step_plain(const Params P, const int* __restrict__ tiles, const Pop fin,
                                                        const Pop fout, float* __restrict__ uout,
                                                        const uint64_t* __restrict__ pres_in,
                                                        uint64_t* __restrict__ pres_out, const int all)
{
    constexpr int NT = TX * TY;
    constexpr int CX = TX + 4, CY = TY + 4;  // phase-field region (halo 2)
    constexpr int RX = TX + 2, RY = TY + 2;  // stress region (halo 1)
    __shared__ float s_ch[kNF][CY][CX];
    __shared__ float s_rho[CY][CX];
    __shared__ float s_txx[RY][RX], s_txy[RY][RX], s_tyy[RY][RX];

    const int lx = threadIdx.x, ly = threadIdx.y, tid = lx + TX * ly;
    const int ntx = (P.nx + TX - 1) / TX;
    const int tile = tiles[blockIdx.x];
    const int around = fluids_around_warp(pres_in, tile, ntx, tid & 31);
    if (!all && one_fluid(around)) return;
    const int x0 = (tile % ntx) * TX, y0 = (tile / ntx) * TY;
    const int nx = P.nx;
    const int N = (int)P.N;
    // pull of the node at (cx, cy) of the phase-field region
    auto pull = [&](int cx, int cy, float q[27]) {
        const int i = (y0 + cy - 2) * nx + (x0 + cx - 2);
        if constexpr (STORE == kStoreF32) {
            const float* b = fin.f + i;
#pragma unroll
            for (int a = 0; a < kQ; a++)
#pragma unroll
                for (int k = 0; k < kNF; k++) q[9 * k + a] = __ldg(b + P.off_pull[k * kQ + a]);
        } else {
            const unsigned short* ob = fin.off + i;
#pragma unroll
            for (int k = 0; k < kNF; k++) {
                float d[kQ];
#pragma unroll
                for (int a = 1; a < kQ; a++) d[a] = dec16<STORE>(__ldg(ob + (8 * k + a - 1) * N));
                q[9 * k] = wq(0) * __ldg(fin.rho + i + k * N) - sum_offsets(d);
#pragma unroll
                for (int a = 1; a < kQ; a++)
                    q[9 * k + a] = wq(a) * __ldg(fin.rho + i + P.off_pull16[k * kQ + a]) +
                                   dec16<STORE>(__ldg(ob + P.off_pull16o[k * kQ + a]));
            }
        }
    };
    if (around & 8) {
        // all but one fluid as traces: the node's own populations are enough
        float q[27], f[kQ];
        pull(lx + 2, ly + 2, q);
#pragma unroll
        for (int a = 0; a < kQ; a++) f[a] = (q[a] + q[9 + a]) + q[18 + a];
        const int v = collide_calm<STORE>(P, fout, uout, (y0 + ly) * nx + x0 + lx, f, sum9(q), sum9(q + 9), sum9(q + 18), 7);
        const int w = __reduce_or_sync(0xffffffffu, v);
        if (lx == 0) reinterpret_cast<uint8_t*>(pres_out + tile)[ly] = row_byte(w);
        return;
    }
    // the lo words of float-float fields do not exist here
    float(*none)[CY][CX] = nullptr;
    int present = 0;
    constexpr int NRING = CX * CY - TX * TY;
    static_assert(NRING <= NT, "the ring of the halo-2 region must not exceed one node per thread");
    if (tid < NRING) {
        int cx, cy;
        ring_position<TX, TY>(tid, cx, cy);
        float q[27];
        pull(cx, cy, q);
        present |= phase_fields<CX, CY>(false, q, s_ch, none, s_rho, cx, cy);
    }
    float f[kQ], r0, r1, r2;
    {
        float q[27];
        pull(lx + 2, ly + 2, q);
        present |= phase_fields<CX, CY>(false, q, s_ch, none, s_rho, lx + 2, ly + 2);
#pragma unroll
        for (int a = 0; a < kQ; a++) f[a] = (q[a] + q[9 + a]) + q[18 + a];
        r0 = sum9(q);
        r1 = sum9(q + 9);
        r2 = sum9(q + 18);
    }
    const bool mixed = single_fluid_or(present) != 1;

    if (mixed) stress_halo1<TX, TY>(P, s_ch, s_rho, s_txx, s_txy, s_tyy, tid);
    __syncthreads();

    float Fx = 0.0f, Fy = 0.0f, g[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
    if (mixed) {
        div_stress<RX>(s_txx, s_txy, s_tyy, lx + 1, ly + 1, Fx, Fy);
#pragma unroll
        for (int k = 0; k < kNF; k++) grad9_f<CX>(s_ch[k], lx + 2, ly + 2, g[2 * k], g[2 * k + 1]);
    }
    float ux, uy;
    const Recolour rc = collide_node(P, f, r0, r1, r2, Fx, Fy, g, ux, uy);
    const int i = (y0 + ly) * nx + x0 + lx;
    if (uout) {
        uout[i] = ux;
        uout[N + i] = uy;
    }
    store_recoloured<STORE>(P, fout, i, f, rc);
    // what this warp's nodes hold, for the tiles around this one in the next step
    const int w = row_bits(recoloured_bits<STORE>(f, r0, r1, r2, rc), f);
    if (lx == 0) reinterpret_cast<uint8_t*>(pres_out + tile)[ly] = row_byte(w);
}

// ------------------------------------------------------------------------------------------
// tiles of any kind: solids, domain edges, the seam, open sides
// ------------------------------------------------------------------------------------------
// the w-weighted neighbour mean, where a line meets no fluid (out of line: rarely called)
template <int STORE>
__device__ __noinline__ double wet_mean(const Params& P, const Pop& fin, const uint8_t* __restrict__ type, int px, int py,
                                        int k)
{
    const Store<STORE> st(fin, P.N);
    return neighbour_mean(P, st, type, px, py, k);
}

// whether the node at unwrapped (X, Y) is fluid, from the geometry words of a tile where they reach:
// it is at (hx, hy) there
template <int HX, int HY>
__device__ __forceinline__ bool fluid_near(const Params& P, const uint8_t* __restrict__ type, const int (*geo)[HX], int hx,
                                           int hy, int X, int Y)
{
    if ((unsigned)hx < (unsigned)HX && (unsigned)hy < (unsigned)HY) return !(geo[hy][hx] & (kGeoSolid | kGeoGhost));
    return node_is_fluid<Store<kStoreF32>>(P, type, X, Y);
}

// Where the line from (px, py) along (dx, dy) first crosses a grid line between two fluid nodes,
// found in single precision: true with the crossed line (vertical x = X or horizontal y = Y) and the
// node below or left of the crossing (ax, ay).  Every decision up to there -- which line comes
// first, between which nodes -- has to be clear by a margin of kRayMargin, some twenty times the
// rounding of the positions (up to 16 long, directions rounded to 6e-8) and a hundred times
// kRayEps; otherwise false, and the double-precision march decides.  (hx, hy): the place of (px, py)
// in the tile's geometry words.
constexpr float kRayMargin = 1e-4f;
template <int HX, int HY>
__device__ __forceinline__ bool float_crossing(const Params& P, const uint8_t* __restrict__ type, const int (*geo)[HX], int hx,
                                               int hy, int px, int py, float dx, float dy, bool& vertical, int& ax,
                                               int& ay)
{
    const float adx = fabsf(dx), ady = fabsf(dy);
    if (!(fminf(adx, ady) >= kRayMargin)) return false;
    const int sx = dx > 0.0f ? 1 : -1, sy = dy > 0.0f ? 1 : -1;
    const float ix = __fdividef(1.0f, adx), iy = __fdividef(1.0f, ady);
    int m = 1, n = 1;  // the next vertical and horizontal grid line, counted from the node
#pragma unroll 1
    for (int it = 0; it < 64; it++) {
        const float tX = m * ix, tY = n * iy;
        const float t = fminf(tX, tY);
        if (t > (float)kRayTmax - 0.01f || fabsf(tX - tY) < kRayMargin) return false;
        vertical = tX < tY;
        // position along the crossed line, relative to the node
        const float r = vertical ? t * dy : t * dx;
        const float rf = floorf(r), fr = r - rf;
        if (fr < kRayMargin || fr > 1.0f - kRayMargin) return false;
        const int fl = (int)rf, rx = vertical ? m * sx : fl, ry = vertical ? fl : n * sy;
        if (fluid_near<HX, HY>(P, type, geo, hx + rx, hy + ry, px + rx, py + ry) &&
            fluid_near<HX, HY>(P, type, geo, hx + rx + !vertical, hy + ry + vertical, px + rx + !vertical,
                               py + ry + vertical)) {
            ax = px + rx;
            ay = py + ry;
            return true;
        }
        if (vertical) m++; else n++;
    }
    return false;
}

// The line of one side of the C_SB node of entry en (normal n) for the local angle th, into its lane.
// The search is done in single precision where that is safe, the crossing itself with the
// expressions of characteristic_line.  geo: the tile's geometry words (or null).
template <int TX, int TY>
__device__ __forceinline__ void wet_line(const Params& P, const TileSet& T, const int (*geo)[TX + 6], const int4 en,
                                         const double2 n, double th, int side, WetLane& c)
{
    constexpr int HX = TX + 6, HY = TY + 6;
    const int node = en.x, px = node % P.nx, py = node / P.nx;
    const int hx = (en.z & 255) + 1, hy = (en.z >> 8 & 255) + 1;  // where the geometry words have the node
    const double dev = fabs(90.0 - th);
    const double phi = dev < kPhiSnap ? 0.0 : dev * (M_PI / 180.0);
    double sn, cs;
    sincos(phi, &sn, &cs);
    if (side) sn = -sn;
    // the line makes the angle phi with n_s (tangent (-n_y, n_x))
    const double dx = fma(cs, n.x, -__dmul_rn(sn, n.y)), dy = fma(cs, n.y, __dmul_rn(sn, n.x));
    Crossing cr{0, 0, 0, 0, 0, 0.0};
    bool vertical;
    if (float_crossing<HX, HY>(P, T.type, geo, geo ? hx : 1 << 30, hy, px, py, (float)dx, (float)dy, vertical, cr.ax,
                               cr.ay)) {
        cr.kind = 2;
        cr.bx = cr.ax + !vertical;
        cr.by = cr.ay + vertical;
        // without fused multiply-add, as characteristic_line
        const double t = (double)(vertical ? cr.ax - px : cr.ay - py) / (vertical ? dx : dy);
        const double s = __dadd_rn((double)(vertical ? py : px), __dmul_rn(t, vertical ? dy : dx));
        cr.fr = s - (double)(vertical ? cr.ay : cr.ax);
    } else {
        cr = characteristic_line<Store<kStoreF32>>(P, T.type, px, py, dx, dy);
    }
    c.fr = cr.fr;
    c.ia = c.ib = -1;
    c.fa = c.fb = 0;
    auto bracket = [&](int X, int Y, int& idx, int& fl) {
        wet_node(P, T.nflag, X, Y, idx, fl);
        const int gx = hx + X - px, gy = hy + Y - py;
        if (gx >= 3 - kNearHalo && gx <= HX - 4 + kNearHalo && gy >= 3 - kNearHalo && gy <= HY - 4 + kNearHalo)
            fl |= kNodeNear;
    };
    if (cr.kind >= 1) bracket(cr.ax, cr.ay, c.ia, c.fa);
    if (cr.kind == 2) bracket(cr.bx, cr.by, c.ib, c.fb);
}

// Threads of a block: one for every node of a tile's halo-2 region (432 of 512), so that each phase
// of a tile is one pass: with 256, which pulled the tile's nodes and the ring around it in turn, a
// tile took 13000 cycles instead of the sum of its memory latencies.
constexpr int kTileThreads = 512;
constexpr int kNoTile = -2;
constexpr int kWetNodes = kTileThreads / 8;  // C_SB nodes wetted at a time

template <int TX, int TY>
struct TileShared {
    static constexpr int HX = TX + 6, HY = TY + 6;  // geometry region (halo 3)
    static constexpr int CX = TX + 4, CY = TY + 4;  // phase-field region (halo 2)
    static constexpr int RX = TX + 2, RY = TY + 2;  // stress region (halo 1)
    int geo[HY][HX];
    float ch[kNF][CY][CX], cl[kNF][CY][CX];  // C_k = hi + lo
    float rho[CY][CX];
    float txx[RY][RX], txy[RY][RX], tyy[RY][RX];
    int4 went[kWetNodes];         // the C_SB nodes of a pass,
    double2 nrm[kWetNodes];       // their normals,
    double raw[kWetNodes][2];     // Eq.(22)'s values of the wetted fluids there, before the limits,
    double wv[kNF][kWetNodes];    // and the three wall values
    double th[2 * kWetNodes];     // angles whose lines have to be looked for,
    short list[2 * kWetNodes];    // and of which node x 2 + fluid
    int wall, flags, todo;        // what the C_SB nodes hold, the fluids present, the list's length
};

// the same finite number, compared as words (a comparison of doubles is one of their slow instructions)
__device__ __forceinline__ bool same_number(double a, double b)
{
    const long long x = __double_as_longlong(a);
    return x == __double_as_longlong(b) && (x & 0x7ff0000000000000LL) != 0x7ff0000000000000LL;
}

// The lines of the next step for the m C_SB nodes of a pass (entries e0 ..), whose wall values of
// this step are in S.wv: Eq.(21), and where its angle changed, the march.  By nt threads (t: this
// one's number), whole warps; nothing of this step waits for it, so two warps that have no node of
// the region do it while the others go on.  The nodes whose angle changed are packed first: an SM
// issues a double-precision warp instruction in some twenty to thirty cycles, and with all lanes
// marching before the wetting, a wall tile took 14 us for it.
template <int TX, int TY>
__device__ __forceinline__ void wet_look(const Params& P, const TileSet& T, int e0, int m, int t, int nt, int bar,
                                         TileShared<TX, TY>& S, int* count)
{
    if (t == 0) *count = 0;
    group_sync(bar, nt);
#pragma unroll 1
    for (int j0 = 0; j0 < 2 * m; j0 += nt) {
        const int j = j0 + t, n = j >> 1, k = j & 1;
        bool turned = false;
        double th = 0.0;
        if (j < 2 * m) {
            const int w = S.went[n].y;
            WetLane* const c = T.cache + (4 * (long long)(e0 + n) + 2 * k);
            const double wm = S.wv[2][n], wl = S.wv[1 - k][n];  // the weights of Eq.(21) for fluid k
            const double om = c[0].wm, ol = c[0].wl, oth = c[0].th;
            const float t_rg = T.wang[3 * w], t_x = T.wang[3 * w + (k == 0 ? 1 : 2)];
            if (!(same_number(om, wm) && same_number(ol, wl))) {
                const double a = 180.0 - (k == 0 ? t_x : t_rg);  // an angle seen from the other side
                th = local_angle(wm, k == 0 ? a : (double)t_x, wl, k == 0 ? (double)t_rg : a);
                c[0].wm = wm;
                c[0].wl = wl;
                // the same angle as when these lanes last marched: the same lines, the same crossings
                turned = !same_number(oth, th);
            }
        }
        const unsigned votes = __ballot_sync(0xffffffffu, turned);
        int at = 0;
        if ((t & 31) == 0 && votes) at = atomicAdd(count, __popc(votes));
        at = __shfl_sync(0xffffffffu, at, 0) + __popc(votes & ((1u << (t & 31)) - 1));
        if (turned) {
            S.list[at] = (short)j;
            S.th[at] = th;
        }
    }
    group_sync(bar, nt);
#pragma unroll 1
    for (int i = t; i < 2 * *count; i += nt) {
        const int j = S.list[i >> 1], n = j >> 1, k = j & 1, side = i & 1;
        WetLane* const c = T.cache + (4 * (long long)(e0 + n) + 2 * k + side);
        WetLane d;
        d.th = S.th[i >> 1];
        wet_line<TX, TY>(P, T, S.geo, S.went[n], S.nrm[n], d.th, side, d);
        c->th = d.th;
        c->fr = d.fr;
        *reinterpret_cast<int4*>(&c->ia) = make_int4(d.ia, d.fa, d.ib, d.fb);
    }
}

// Wetting of the C_SB nodes of a tile's phase-field region (entries e0 .. e0 + cnt of the set's
// list): C at the nodes that bracket the crossings of the two characteristic lines of the two wetted
// fluids, which the last step looked for (wet_look), and Eq.(22).  Eight lanes per node -- lane =
// 4 k + 2 side + end -- pull one of the up to two nodes of a line each.  The values go to the region's
// phase fields (rho := 1 there), to S.wv and, for the nodes that the tile owns, to cw_out.  A node
// near several tiles is wetted by each of them, with the same result: 1.6 times the work of a pass
// over the nodes, but no launch that the tiles have to wait for.  one: the fluids around where all that
// can reach the region is calm, else 7; where that is one, the nodes near the region hold it alone and
// with a positive density (C_k exactly 1 or 0), and need no pull.  Returns the
// fluids with a nonzero wall value (bit k), in bit 3 whether some node's values are mixed, in bit 4
// whether a line ends in a node that is not near, and in bit 5 whether some value of a fluid other than
// calm - 1 is more than a trace.
template <int TX, int TY, int STORE>
__device__ __forceinline__ int wet_entries(const Params& P, const TileSet& T, int e0, int cnt, int one,
                                           int calm, const Pop& fin, double* cw_out, TileShared<TX, TY>& S)
{
    const long long N = P.N;
    const int tid = threadIdx.x;
    int bits = 0;
#pragma unroll 1
    for (int b0 = 0; b0 < cnt; b0 += kWetNodes) {
        const int m = min(cnt - b0, kWetNodes);  // nodes of this pass
        if (b0 > 0) {
            // the pass before: its lines of the next step, then this one's nodes in its place
            __syncthreads();
            wet_look<TX, TY>(P, T, e0 + b0 - kWetNodes, kWetNodes, tid, kTileThreads, 0, S, &S.flags);
            __syncthreads();
            if (tid < m) {
                S.went[tid] = T.went[e0 + b0 + tid];
                S.nrm[tid] = T.wnrm[e0 + b0 + tid];
            }
            if (tid == 0) S.flags = 0;
            __syncthreads();
        }
        if ((tid & ~31) < 8 * m) {
            const bool valid = tid < 8 * m;
            const int end = tid & 1, side = tid >> 1 & 1, k = tid >> 2 & 1;
            const int e = valid ? tid >> 3 : 0;
            const WetLane c = T.cache[4 * (long long)(e0 + b0 + e) + 2 * k + side];
            double v = 0.0;
            if (valid) {
                const int4 en = S.went[e];
                const int idx = end ? c.ib : c.ia, fl = end ? c.fb : c.fa, node = en.x;
                if (idx >= 0 ? !(fl & kNodeNear) : end == 0) bits |= 16;
                if (idx >= 0 && (fl & kNodeNear) && __popc((unsigned)one) == 1)
                    v = one >> relabel(k, en.z & kWetPar) & 1 ? 1.0 : 0.0;  // in the tile's frame
                else if (idx >= 0)
                    v = wet_fraction<STORE>(P, fin, idx, fl, k);
                else if (end == 0)
                    v = wet_mean<STORE>(P, fin, T.type, node % P.nx, node / P.nx, k);
            }
            const double o = __shfl_xor_sync(0xffffffffu, v, 1);
            const double ca = end ? o : v, cb = end ? v : o;
            double cd = ca;
            if (c.ib >= 0 && !same_number(ca, cb)) cd = ca + c.fr * (cb - ca);
            // Eq.(22): max of the two lines for theta_k <= 90 deg, min otherwise
            const double other = __shfl_xor_sync(0xffffffffu, cd, 2);
            double cp = cd;
            if (!same_number(cd, other))
                cp = c.th <= 90.0 ? fmax(cd, other) : fmin(cd, other);
            if (valid && (tid & 3) == 0) S.raw[e][k] = cp;
        }
        __syncthreads();
        if (tid < m) {
            double c0 = S.raw[tid][0], c1 = S.raw[tid][1], c2;
            const bool z0 = same_number(c0, 0.0), z1 = same_number(c1, 0.0);
            // one fluid at the node: no double-precision instructions
            const bool pure = (z0 && z1) || (z0 && same_number(c1, 1.0)) || (z1 && same_number(c0, 1.0));
            if (pure) {
                c2 = z0 && z1 ? 1.0 : 0.0;
            } else {
                // fractions stay in [0, 1] (a no-op unless 16-bit storage rounded a density below 0)
                c0 = fmin(fmax(c0, 0.0), 1.0);
                c1 = fmin(fmax(c1, 0.0), 1.0);
                const double s = c0 + c1;
                if (s > 1.0) {
                    c0 /= s;
                    c1 /= s;
                }
                c2 = fmax(0.0, 1.0 - c0 - c1);
            }
            S.wv[0][tid] = c0;
            S.wv[1][tid] = c1;
            S.wv[2][tid] = c2;
            const int4 en = S.went[tid];
            if (en.z & kWetOwner) {
                cw_out[en.x] = c0;
                cw_out[N + en.x] = c1;
                cw_out[2 * N + en.x] = c2;
            }
            // FP64 split into hi + lo, relabelled across a modified periodic seam
            const int cx = en.z & 255, cy = en.z >> 8 & 255;
            const bool par = en.z & kWetPar;
            const double cc[kNF] = {par ? c2 : c0, c1, par ? c0 : c2};
#pragma unroll
            for (int j = 0; j < kNF; j++) {
                float h, l = 0.0f;
                if (pure) {
                    h = same_number(cc[j], 0.0) ? 0.0f : 1.0f;
                } else {
                    h = (float)cc[j];
                    l = (float)(cc[j] - (double)h);
                }
                S.ch[j][cy][cx] = h;
                S.cl[j][cy][cx] = l;
                if (!same_number(cc[j], 0.0)) bits |= 1 << j;
                if (j + 1 != calm && !(h <= kCalmWall)) bits |= 32;
            }
            S.rho[cy][cx] = 1.0f;
            if (!pure && fmax(fmax(c0, c1), c2) < 1.0 - kMixEps) bits |= 8;
        }
    }
    return bits;
}

// the lines of the current wall values Cw, for every entry of the set (after the state or the wall
// angles were replaced): what wet_look does at the end of a step
__global__ void k_wet_look(const Params P, const TileSet T, const int n, const double* __restrict__ Cw)
{
    const int j = blockIdx.x * blockDim.x + threadIdx.x;
    if (j >= 4 * n) return;
    const int4 en = T.went[j >> 2];
    const int side = j & 1, k = j >> 1 & 1;
    const double wm = Cw[2 * P.N + en.x], wl = Cw[(1 - k) * P.N + en.x];
    const float t_rg = T.wang[3 * en.y], t_x = T.wang[3 * en.y + (k == 0 ? 1 : 2)];
    WetLane d;
    d.wm = wm;
    d.wl = wl;
    d.th = k == 0 ? local_angle(wm, 180.0 - t_x, wl, t_rg) : local_angle(wm, t_x, wl, 180.0 - t_rg);
    wet_line<kTX, kTY>(P, T, nullptr, en, T.wnrm[j >> 2], d.th, side, d);
    T.cache[j] = d;
}

// initial wall values: w-weighted mean of the fluid neighbours, for each fluid
template <class S>
__global__ void k_wet_init(const Params P, const int nw, const int* __restrict__ widx, const S st,
                           const uint8_t* __restrict__ type, double* __restrict__ Cw)
{
    const int w = blockIdx.x * blockDim.x + threadIdx.x;
    if (w >= nw) return;
    const int i = widx[w];
    const int px = i % P.nx, py = i / P.nx;
    for (int k = 0; k < kNF; k++) {
        Cw[k * P.N + i] = neighbour_mean(P, st, type, px, py, k);
    }
}

// Programmatic dependent launch (nothing happens in a launch without it): let the next kernel of the
// stream start its blocks where there is room; wait until the kernels before have ended and their
// writes can be read.
__device__ __forceinline__ void launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void wait_prerequisites() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

// fluids_around for the tiles of a record (this lane's entry of the list: nbr; own: the tile's word)
__device__ __forceinline__ int fluids_reaching(const uint64_t* __restrict__ pres, int nbr, uint64_t own)
{
    int around = nbr == -1 ? 7 : 0;  // an open column: any fluid
    bool calm = nbr < -1;
    if (nbr >= 0) {
        const uint64_t b = pres[nbr >> 1];
        const int v = word_fluids(b), d1 = word_calm(own);
        const bool seam = nbr & 1;  // across it fluids 0 and 2 swap
        around = seam ? (v & 2) | (v & 1) << 2 | v >> 2 : v;
        calm = word_calm_in(b, seam && d1 > 0 ? 4 - d1 : d1);
    }
    around = __reduce_or_sync(0xffffffffu, around);
    return around | (__all_sync(0xffffffffu, calm) ? 8 : 0);
}

// Bits 5-6 of a tile's word (at most 2): for how many steps the wall values of every C_SB node that the
// tile sees have been those of the one fluid around it alone, with lines that end in nodes near it.
// After two both arrays of wall values hold them, and while the tiles around keep holding that fluid
// alone, and calm, nothing of the wetting changes.  (The tile itself is among those, and has a fluid node, so it
// is the same fluid.)
__device__ __forceinline__ int settled_steps(uint64_t word, int around)
{
    return __popc((unsigned)around & 7u) == 1 ? (int)(word >> 5 & 3) : 0;
}
// a tile that needs no wetting and holds one fluid after the pull: k_step_one's (calm around, bit 3: a
// density that became zero or NaN there would reach the wall values in this step)
__device__ __forceinline__ bool settled_single(int around, int cnt, uint64_t word)
{
    return __popc((unsigned)around & 7u) == 1 && (cnt == 0 || ((around & 8) && settled_steps(word, around) == 2));
}

// One step of tile T.rec[blockIdx.x] (any kind): thread t < TX TY has the tile's node t, the next ones a
// node of the ring that the halo-2 region has around it.
//   geometry words of the halo-3 region into shared memory
//   wetting of the C_SB nodes of the phase-field region
//   one fluid around (the words of the tiles that the halo-3 region touches, and the wall values):
//     9 populations per own node as in k_step_one
//   all but one fluid as traces (calm_bits): the own nodes' populations, no gradients
//   else the pulls, phase fields, stress, force, collision and recolouring of all three fluids;
//     where a C_SB node of the region has mixed wall values (a contact line at or near it) the
//     phase fields are float-float, decided anew every step
// What bounds it: on small grids the chain of memory latencies (about 700 cycles each) and instruction
// cache misses (6 of its stalls per issued instruction on 128 x 64) in a wall tile, 18000 cycles of
// which the wetting is 8500; so what is known early is loaded early: the tile's record in one load,
// all that hangs on it in the next.  It takes the place of a wetting pass and two launches behind it:
// a step of 128 x 64 took 17.5 us instead of 27.6, of 320 x 180 17.2 instead of 27.9, of the 800 x 375
// pillars 28.6 instead of 35.5, and of the 4096 x 2048 ones 223 instead of 240 (with what came after --
// one launch per step, calm tiles -- now 15.5, 16.7, 20 and 160 after some hundred steps).
// (Measured and left out: many steps in one cooperative launch whose blocks wait for one another, 14 to
// 80 us where this took 12 to 44; the region's populations copied to shared memory during the wetting,
// no gain; 256 threads a tile, each with two nodes of the region in turn, 1.5 times slower.)
template <int TX, int TY, int STORE>
__global__ void __launch_bounds__(kTileThreads, 2) k_tile(const Params P, const TileSet T, const Pop fin, const Pop fout,
                                                          double* cw_out, float* uout, const uint64_t* pres_in,
                                                          uint64_t* pres_out, const int full_write, const int one)
{
    using TS = TileShared<TX, TY>;
    constexpr int NT = kTileThreads, CX = TS::CX, CY = TS::CY, RX = TS::RX, RY = TS::RY, HX = TS::HX, HY = TS::HY;
    constexpr int NOWN = TX * TY, NC = CX * CY, NR = RX * RY;
    static_assert(TX == 32 && TY == 8 && NC <= NT, "one warp per row, one node of the region per thread");
    // the warps that have a node of the region; the others look for the lines of the next step
    constexpr int NB = (NC + 31) / 32 * 32;
    static_assert(NT - NB >= 32, "a warp for the lines");
    __shared__ TS S;
    const int tid = threadIdx.x, lane = tid & 31;
    const int N = (int)P.N;
    const int word32 = T.rec[blockIdx.x * kTileRecInts + lane];  // one word of the record per lane
    const int tile = __shfl_sync(0xffffffffu, word32, 0), e0 = __shfl_sync(0xffffffffu, word32, 1),
              cnt = __shfl_sync(0xffffffffu, word32, 2);
    const int nbr = lane >= kTileRecHead ? word32 : kNoTile;
    const int ntx = (P.nx + TX - 1) / TX;
    const int x0 = (tile % ntx) * TX, y0 = (tile / ntx) * TY;
    // fluids stored in the tiles that reach the region (every warp for itself), and whether the
    // tile's wall values have settled
    int around;
    uint64_t mine;
    launch_dependents();
    if (one) {
        wait_prerequisites();
        mine = pres_in[tile];
        around = fluids_reaching(pres_in, nbr, mine);
        if (settled_single(around, cnt, mine)) return;  // k_step_one's
    }
    for (int j = tid; j < HX * HY; j += NT) {
        const int hx = j % HX, hy = j / HX;
        S.geo[hy][hx] = geo_word(P, T.type, x0 + hx - 3, y0 + hy - 3);
    }
    if (tid < min(cnt, kWetNodes)) {
        S.went[tid] = T.went[e0 + tid];
        S.nrm[tid] = T.wnrm[e0 + tid];
    }
    if (tid == 0) S.wall = S.flags = 0;
    if (!one) {
        wait_prerequisites();  // up to here nothing that a step writes was read
        mine = pres_in[tile];
        around = fluids_reaching(pres_in, nbr, mine);
    }
    bool calm = around & 8;
    around &= 7;
    const bool inside = tid < NOWN;  // a node of the tile itself, row tid / 32 (one warp)
    uint8_t* const word = reinterpret_cast<uint8_t*>(pres_out + tile) + (tid >> 5);
    const int old = !inside || full_write ? 7 : *word & 7;  // what this row of the output buffer still holds
    __syncthreads();

    // this thread's position in the phase-field region
    int cx = 0, cy = 0;
    if (inside) {
        cx = lane + 2;
        cy = (tid >> 5) + 2;
    } else if (tid < NC) {
        ring_position<TX, TY>(tid - NOWN, cx, cy);
    }
    int hx = cx + 1, hy = cy + 1;
    int own = tid < NC ? S.geo[hy][hx] : kGeoSolid;
    const bool own_fluid = inside && !(own & kGeoSolid) && x0 + cx - 2 < P.nx && y0 + cy - 2 < P.ny;
    int px = hx;
    if (own & kGeoGhost) {
        // beyond an open side: the boundary-column node (zero gradient)
        const int X = x0 + hx - 3;
        px += X < 0 ? -X : P.nx - 1 - X;
    }
    bool df = false;
    int wp = 0;
    if (cnt > 0) {
        const int b = __reduce_or_sync(
            0xffffffffu, wet_entries<TX, TY, STORE>(P, T, e0, cnt, calm ? around : 7, word_calm(mine), fin, cw_out, S));
        if (lane == 0 && b) atomicOr(&S.wall, b);
        __syncthreads();
        df = S.wall & 8;
        wp = S.wall & 7;
        calm = calm && !(S.wall & 40);
    }
    // steps in a row in which one fluid was around and every wall value and line was that fluid's
    const int quiet = cnt > 0 && S.wall == around ? min(settled_steps(mine, around) + 1, 2) : 0;
    if (tid >= NB) {
        if (cnt > 0) {
            const int last = (cnt - 1) / kWetNodes * kWetNodes;
            wet_look<TX, TY>(P, T, e0 + last, cnt - last, tid - NB, NT - NB, 2, S, &S.todo);
        }
        return;
    }
    if (!df && __popc((unsigned)(around | wp)) == 1) {
        // ---- one fluid: as in k_step_one ----
        if (!inside) return;
        const int k = __ffs(around | wp) - 1, i = own & kGeoIdx;
        bool plain = true, still = true;
        float f[kQ], r = 1.0f, ux = 0.0f, uy = 0.0f;
        if (own_fluid) {
#pragma unroll
            for (int a = 0; a < kQ; a++) {
                const int g = S.geo[hy - ey(a)][hx - ex(a)];
                const bool bb = g & kGeoSolid;
                const int s = bb ? own : g;
                load_fluid<STORE>(P, fin, s & kGeoIdx, bb ? opp(a) : a, (s & kGeoPar) && k != 1 ? 2 - k : k, f[a]);
            }
            r = sum9(f);
            plain = collide_single(P, k, f, r, ux, uy);
            still = calm_bits<STORE>(f, r, 0.0f, 0.0f, 0.0f) == 0;
        }
        const bool all = all_single(plain, still, f);
        if (own_fluid) {
            if (uout) {
                uout[i] = ux;
                uout[N + i] = uy;
            }
            const int write = all ? old | 1 << k : 7;
#pragma unroll 1
            for (int l = 0; l < kNF; l++) {
                if (!(write & (1 << l))) continue;
                const float c = plain ? (l == k ? 1.0f : 0.0f) : fraction(l == k ? r : 0.0f, r);
                store_fluid<STORE>(P, fout, l, i, f, c);
            }
        }
        const unsigned some = __ballot_sync(0xffffffffu, own_fluid);
        if (lane == 0)
            *word = (uint8_t)((some ? (all ? 1 << k | (still ? (k + 1) << 3 : 0) : 7) : 0) | (tid == 0 ? quiet << 5 : 0));
        return;
    }
    if (calm) {
        // ---- several fluids, all but one as traces: no gradients (calm_bits) ----
        if (!inside) return;
        int bits = 0;
        if (own_fluid) {
            float f[kQ], r[kNF] = {0.0f, 0.0f, 0.0f};
#pragma unroll
            for (int a = 0; a < kQ; a++) f[a] = 0.0f;
#pragma unroll
            for (int k = 0; k < kNF; k++) {
                if (!(around >> k & 1)) continue;
                float q[kQ];
#pragma unroll
                for (int a = 0; a < kQ; a++) {
                    const int g = S.geo[hy - ey(a)][hx - ex(a)];
                    const bool bb = g & kGeoSolid;
                    const int s = bb ? own : g;
                    load_fluid<STORE>(P, fin, s & kGeoIdx, bb ? opp(a) : a, (s & kGeoPar) && k != 1 ? 2 - k : k, q[a]);
                }
                r[k] = sum9(q);
#pragma unroll
                for (int a = 0; a < kQ; a++) f[a] = f[a] + q[a];
            }
            bits = collide_calm<STORE>(P, fout, uout, own & kGeoIdx, f, r[0], r[1], r[2], old | around);
        }
        const int v = __reduce_or_sync(0xffffffffu, bits);
        if (lane == 0) *word = row_byte(v);
        return;
    }

    // ---- pulls, densities and phase fields of the halo-2 region ----
    int present = wp;
    float f[kQ], r0 = 0.0f, r1 = 0.0f, r2 = 0.0f;
    if (!(own & kGeoSolid)) {
        own = S.geo[hy][px];
        hx = px;
        float q[27];
        bool open = false;
#pragma unroll
        for (int a = 0; a < kQ; a++) {
            const int g = S.geo[hy - ey(a)][hx - ex(a)];
            const bool bb = g & kGeoSolid;
            const int s = bb ? own : g;
            load_direction<STORE>(P, fin, s & kGeoIdx, bb ? opp(a) : a, q + a);
        }
#pragma unroll
        for (int a = 1; a < kQ; a++) {
            const int g = S.geo[hy - ey(a)][hx - ex(a)];
            if ((g & kGeoSolid ? own : g) & kGeoPar) {
                const float t = q[a];
                q[a] = q[18 + a];
                q[18 + a] = t;
            }
            if (g & kGeoGhost) {
                open = true;
                q[a] = q[9 + a] = q[18 + a] = 0.0f;
            }
        }
        if (own & kGeoPar) {
            const float t = q[0];
            q[0] = q[18];
            q[18] = t;
        }
        if (open) zou_he(P, q, x0 + hx - 3 == 0);
        present |= phase_fields<CX, CY>(df, q, S.ch, S.cl, S.rho, cx, cy);
#pragma unroll
        for (int a = 0; a < kQ; a++) f[a] = (q[a] + q[9 + a]) + q[18 + a];
        r0 = sum9(q);
        r1 = sum9(q + 9);
        r2 = sum9(q + 18);
    } else if (geo_class(own) == kSI && tid < NC) {
#pragma unroll
        for (int k = 0; k < kNF; k++) S.ch[k][cy][cx] = S.cl[k][cy][cx] = 0.0f;
        S.rho[cy][cx] = 0.0f;
    }
    {
        const int pw = __reduce_or_sync(0xffffffffu, present);
        if (lane == 0 && pw) atomicOr(&S.flags, pw);
    }
    group_sync(1, NB);
    const bool mixed = __popc((unsigned)(S.flags & 7)) != 1;

    // ---- stress tensor of Eq.(10) on the halo-1 region; gradients of the own nodes ----
    float Fx = 0.0f, Fy = 0.0f, gr[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
    if (mixed) {
        if (tid < NR) {
            int rx = cx - 1, ry = cy - 1;
            if (!inside) {
                // the ring of the halo-1 region: two rows, then two columns
                const int j = tid - NOWN;
                ry = j < 2 * RX ? (j < RX ? 0 : RY - 1) : 1 + (j - 2 * RX) / 2;
                rx = j < 2 * RX ? j % RX : ((j - 2 * RX) & 1 ? RX - 1 : 0);
            }
            float Txx, Txy, Tyy, gxk[kNF], gyk[kNF];
            stress_at<HX, CX, CY>(P, S.geo, S.ch, S.cl, S.rho, df, rx, ry, gxk, gyk, Txx, Txy, Tyy);
            S.txx[ry][rx] = Txx;
            S.txy[ry][rx] = Txy;
            S.tyy[ry][rx] = Tyy;
#pragma unroll
            for (int k = 0; k < kNF; k++) {
                gr[2 * k] = gxk[k];
                gr[2 * k + 1] = gyk[k];
            }
        }
        group_sync(1, NB);
        if (own_fluid) div_stress<RX>(S.txx, S.txy, S.tyy, cx - 1, cy - 1, Fx, Fy);
    }
    // ---- velocity, MRT collision with forcing, recolouring, stores ----
    if (!inside) return;
    int bits = 0;
    if (own_fluid) {
        const int i = own & kGeoIdx;
        float ux, uy;
        const Recolour rc = collide_node(P, f, r0, r1, r2, Fx, Fy, gr, ux, uy);
        if (uout) {
            uout[i] = ux;
            uout[N + i] = uy;
        }
        store_recoloured<STORE>(P, fout, i, f, rc);
        bits = recoloured_bits<STORE>(f, r0, r1, r2, rc);
    }
    // what this row's fluid nodes hold, for the tiles around in the next step
    const int v = row_bits(bits, f);
    if (lane == 0) *word = row_byte(v);
}

// Pure tiles around which the step's input holds one fluid k (pres_in): k alone is in the tile
// after the pull (a fluid absent from all of a node's sources stays absent, and the recolouring
// keeps it at zero), so 9 populations per node are pulled, collided and written: 72 B per node
// (40 B in the 16-bit storage) instead of 216 (120).  The other fluids' planes have to read as
// zeros to whoever reads all 27 there, and do without being written: pres_out[tile] still
// describes the output buffer as it was written two steps ago, and only a fluid that it names in a
// row is cleared there, once.  So the planes of a fluid that a tile's word does not name are zeros
// in that buffer.  (full_write: the output is not the buffer that pres_out described, so they are
// cleared always.)  The other pure tiles are left to the kernels that move all 27 planes.
//
// The tiles near solids or the domain edge in which nothing of the wetting changes (settled_single) are
// done the same way, with the flags of each node (directions that bounce back, wraps) in place of fixed
// offsets.
//
// A warp takes kOneRows rows of 32 nodes, two in flight: nothing is shared between threads, each
// population is read once, and the loads of a warp are whole lines but for the shift by one node in x.
// It is bound by HBM: alone on the 4096 x 2048 pillars 85 us for 547 MB, the rate of a copy, at some 310
// instructions a row with the tile's look-up (12.2 M for the 39,000 rows of the 2048 x 1024 ones after 1500
// steps; 68 more with lane-wise plane addresses) and 62 % issue, so what counts is warps in flight: no shared
// memory, no barriers, 40 registers in every storage.  (Two rows per thread in packed single-precision
// instructions, with 62 registers: 158 us a step instead of 156.)  On the 4096 x 2048 pillars, where 93 % of
// the pure tiles are such after 200 steps, the pure tiles took 338 us a step (FP16: 410) in the kernels that
// move all 27 planes; the whole step, all kernels, takes 160 us with this one (FP16: 162).  (Inside the ring
// kernel, with 9-plane boxes, the same tiles took 1200 cycles of a consumer group and 1500 of its one
// producer each: 270 us.)
constexpr int kOneThreads = 128;
// rows of a pure tile per warp (a tile near solids: 1, there are few of them and each row waits for its
// flags first); 8, 4 and 2 rows: 180, 175 and 182 us a step of the 4096 x 2048 pillars
constexpr int kOneRows = 4;
template <int TX, int TY, int STORE, bool PURE>
__global__ void __launch_bounds__(kOneThreads) k_step_one(const Params P, const TileSet T, const int* __restrict__ tiles,
                                                          const int ntiles, const Pop fin, const Pop fout,
                                                          float* __restrict__ uout,
                                                          const uint64_t* __restrict__ pres_in,
                                                          uint64_t* __restrict__ pres_out, const int full_write)
{
    static_assert(TX == 32 && TY == 8, "a row per warp instruction, one byte of the tile's word per row");
    constexpr int RW = PURE ? kOneRows : 1;  // rows of a warp
    const int u = blockIdx.x * (kOneThreads / 32) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
    const int w = u / (TY / RW), row0 = u % (TY / RW) * RW;
    if (w >= (PURE ? ntiles : T.ntiles)) return;
    const int ntx = (P.nx + TX - 1) / TX;
    int tile, around;
    uint64_t word = 0;
    if constexpr (PURE) {
        // one lane per tile around; what a warp reduction returns is uniform to the compiler, which
        // then addresses the planes by uniform registers
        tile = __reduce_or_sync(0xffffffffu, tiles[w]);
        int v = 0;
        if (lane < 9) v = word_fluids(pres_in[tile + (lane / 3 - 1) * ntx + lane % 3 - 1]);
        around = __reduce_or_sync(0xffffffffu, v);
        if (__popc((unsigned)around) != 1) return;
    } else {
        const int r = T.rec[w * kTileRecInts + lane];
        tile = __shfl_sync(0xffffffffu, r, 0);
        const int cnt = __shfl_sync(0xffffffffu, r, 2);
        const uint64_t mine = pres_in[tile];
        around = fluids_reaching(pres_in, lane >= kTileRecHead ? r : kNoTile, mine);
        if (!settled_single(around, cnt, mine)) return;
        around &= 7;
        word = mine & 0x60;  // settled it stays
    }
    if (!PURE && row0 >= P.ny - (tile / ntx) * TY) {
        if (lane == 0) reinterpret_cast<uint8_t*>(pres_out + tile)[row0] = 0;
        return;
    }
    const uint64_t old = full_write ? 0x0707070707070707ull : pres_out[tile];
    const int k = __ffs(around) - 1;
    const int nx = P.nx, N = (int)P.N;
    const int x0 = (tile % ntx) * TX, y0 = (tile / ntx) * TY;
    const int rows = PURE ? row0 + RW : min(row0 + RW, P.ny - y0);
    const bool column = PURE || x0 + lane < nx;
    // the fluid's planes at the tile's corner (FP32 storage)
    const int corner = y0 * nx + x0;
    const float* src[kQ];
    float* dst[kQ];
#pragma unroll
    for (int a = 0; a < kQ; a++) {
        src[a] = fin.f + (corner + k * kQ * N + P.off_pull[a]);
        dst[a] = fout.f + (corner + k * kQ * N + P.off_plane[a]);
    }
#pragma unroll 2
    for (int row = row0; row < rows; row++) {
        const int i = (y0 + row) * nx + x0 + lane;
        float f[kQ];
        bool fluid = true;
        if constexpr (PURE) {
            if constexpr (STORE == kStoreF32) {
                const unsigned o = (unsigned)(row * nx + lane);
#pragma unroll
                for (int a = 0; a < kQ; a++) f[a] = __ldg(src[a] + o);
            } else {
                const float* rb = fin.rho + i + k * N;
                const unsigned short* ob = fin.off + i + 8 * k * N;
                float d[kQ];
#pragma unroll
                for (int a = 1; a < kQ; a++) d[a] = dec16<STORE>(__ldg(ob + (a - 1) * N));
                f[0] = wq(0) * __ldg(rb) - sum_offsets(d);
#pragma unroll
                for (int a = 1; a < kQ; a++)
                    f[a] = wq(a) * __ldg(rb + P.off_pull16[a]) + dec16<STORE>(__ldg(ob + P.off_pull16o[a]));
            }
        } else {
            const int fl = column ? (int)__ldg(T.nflag + i) : kNodeSolid;
            fluid = !(fl & kNodeSolid);
            if (fluid) {
                const int xm = fl & kNodeX0 ? nx - 1 : -1, xp = fl & kNodeXN ? 1 - nx : 1;
                const int ym = fl & kNodeY0 ? (P.ny - 1) * nx : -nx, yp = fl & kNodeYN ? (1 - P.ny) * nx : nx;
#pragma unroll
                for (int a = 0; a < kQ; a++) {
                    const bool bb = a > 0 && (fl >> a & 1);
                    const bool over = (ex(a) == 1 && (fl & kNodeX0)) || (ex(a) == -1 && (fl & kNodeXN));
                    const int d = (ex(a) == 1 ? xm : (ex(a) == -1 ? xp : 0)) + (ey(a) == 1 ? ym : (ey(a) == -1 ? yp : 0));
                    const bool swap = P.bc_x == kModPer && over && !bb && k != 1;
                    load_fluid<STORE>(P, fin, bb ? i : i + d, bb ? opp(a) : a, swap ? 2 - k : k, f[a]);
                }
            }
        }
        float r = 1.0f, ux = 0.0f, uy = 0.0f;
        bool plain = true, still = true;
        if (fluid) {
            r = sum9(f);
            plain = collide_single(P, k, f, r, ux, uy);
            still = calm_bits<STORE>(f, r, 0.0f, 0.0f, 0.0f) == 0;
            // (what all_single does otherwise; with this form the 16-bit storages need 40 registers, not 48)
            if (PURE && !still) plain = plain && all_finite(f);
            if (uout) {
                uout[i] = ux;
                uout[N + i] = uy;
            }
        }
        bool all;
        if constexpr (PURE) {
            all = __all_sync(0xffffffffu, plain);
            still = __all_sync(0xffffffffu, still);
        } else {
            all = all_single(plain, still, f);
        }
        const int rowold = (int)(old >> (8 * row)) & 7;
        // fluids to write: k, and those that this row of the buffer still holds, as zeros; all of
        // them where a density has no fraction
        const int write = all ? rowold | 1 << k : 7;
        if (fluid) {
            if (write == 1 << k) {
                if constexpr (STORE == kStoreF32) {
                    const unsigned o = (unsigned)(row * nx + lane);
#pragma unroll
                    for (int a = 0; a < kQ; a++) dst[a][o] = f[a];
                } else {
                    store_fluid<STORE>(P, fout, k, i, f, 1.0f);
                }
            } else {
#pragma unroll 1
                for (int l = 0; l < kNF; l++) {
                    if (!(write & (1 << l))) continue;
                    const float c = plain ? (l == k ? 1.0f : 0.0f) : fraction(l == k ? r : 0.0f, r);
                    store_fluid<STORE>(P, fout, l, i, f, c);
                }
            }
        }
        const bool some = PURE || __ballot_sync(0xffffffffu, fluid);
        const int byte = some ? (all ? 1 << k | (still ? (k + 1) << 3 : 0) : 7) : 0;
        if (lane == 0)
            reinterpret_cast<uint8_t*>(pres_out + tile)[row] = (uint8_t)(byte | (row == 0 ? (int)word : 0));
    }
}

// Pure FP32 tiles through a ring of bulk tensor copies, warp-specialised: one producer warp and
// two consumer groups of TX x TY threads per block, one block per SM (persistent).  Tile j of the
// block (tiles[blockIdx.x + j gridDim.x]) lands in ring buffer j % 3 -- its 27-plane pull box,
// (TX + 8) x (TY + 6) nodes from (x0 - 4, y0 - 3), by one copy -- and is computed by group j % 2.
// A group releases its buffer as soon as its pulls are done (one arrival per warp on the buffer's
// "empty" barrier), and the producer refills it at once with tile j + 3, so up to three boxes are
// in flight or waiting while the groups compute their force, collision and recolouring.  The
// "full" barrier of tile j is full[j % 6]: its tiles j, j + 6, ... are consumed in order by the
// same group, so a wait never meets a phase two behind (no parity aliasing).  Every wait is
// bounded: a consumer that gives up sets the error bit and its group returns; the producer gives
// up on a buffer that is never released, and before exiting it waits (full limit) for every copy
// it issued, so no copy lands in the shared memory of a later block.  The arithmetic is that of
// k_step_tma and k_step_plain, so the results are identical.
// The tiles with one fluid around are k_step_one's unless all is set; the producer passes over them, 32 at a time
// (each lane looks one up).  Each warp records the fluids its nodes hold (one byte of
// pres_out[tile] per warp), so that the tiles around know in the next step.
constexpr int kRingBufs = 3;
template <int TX, int TY>
__global__ void __launch_bounds__(2 * TX * TY + 32, 1) k_step_ring(const Params P, const int* __restrict__ tiles,
                                                                    const int ntiles, float* __restrict__ fout,
                                                                    float* __restrict__ uout,
                                                                    const __grid_constant__ CUtensorMap tm_in,
                                                                    const uint64_t* __restrict__ pres_in,
                                                                    uint64_t* __restrict__ pres_out, const int all)
{
    constexpr int NT = TX * TY;               // threads of a consumer group
    constexpr int NW = NT / 32;               // warps of a consumer group
    constexpr int CX = TX + 4, CY = TY + 4;  // phase-field region (halo 2)
    constexpr int RX = TX + 2, RY = TY + 2;  // stress region (halo 1)
    constexpr int BX = TX + 8, BY = TY + 6;  // pull-source box
    constexpr int NBOX = kQ * kNF * BY * BX;
    constexpr int NBOXP = (NBOX + 31) / 32 * 32;  // keeps every buffer 128-byte aligned
    constexpr int NRING = CX * CY - TX * TY;
    static_assert(NRING <= NT, "the ring of the halo-2 region must not exceed one node per thread");
    static_assert(NT % 32 == 0, "whole warps per group");
    __shared__ float s_ch[2][kNF][CY][CX];
    __shared__ float s_rho[2][CY][CX];
    __shared__ float s_txx[2][RY][RX], s_txy[2][RY][RX], s_tyy[2][RY][RX];
    __shared__ __align__(8) uint64_t s_full[2 * kRingBufs], s_empty[kRingBufs];
    __shared__ int s_flags[2][2];
    __shared__ int s_tile[2 * kRingBufs];  // by full-barrier slot: the tile
    extern __shared__ unsigned char dsm[];
    float* ring = reinterpret_cast<float*>(dsm + ((128u - (smem_u32(dsm) & 127u)) & 127u));  // [3][27][BY][BX]

    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int ntx = (P.nx + TX - 1) / TX;
    if ((int)blockIdx.x >= ntiles) return;
    const int njobs = (ntiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
    if (threadIdx.x == 0) {
        for (int m = 0; m < 2 * kRingBufs; m++) mbar_init(smem_u32(&s_full[m]), 1);
        for (int b = 0; b < kRingBufs; b++) mbar_init(smem_u32(&s_empty[b]), NW);
        fence_mbar_init();
        s_flags[0][0] = s_flags[0][1] = s_flags[1][0] = s_flags[1][1] = 0;
    }
    __syncthreads();

    // ---------------- producer warp ----------------
    if (warp == 2 * NW) {
        // job j: the tile's box into buffer j % 3, which is free once the group that computed job
        // j - 3 has pulled from it; no copy for tile -1, which ends the group's loop
        auto send = [&](int tile, int j) {
            const int b = j % kRingBufs;
            if (j >= kRingBufs && tile >= 0) {
                bool free = false;
                const uint32_t par = (uint32_t)((j / kRingBufs - 1) & 1);
                for (int it = 0; it < P.wait_polls && !free; it++) free = mbar_try_wait(smem_u32(&s_empty[b]), par);
                if (!free) return false;
            }
            // written before the arrive, whose release the consumers' wait acquires
            s_tile[j % (2 * kRingBufs)] = tile;
            const uint32_t full = smem_u32(&s_full[j % (2 * kRingBufs)]);
            if (tile < 0) {
                mbar_arrive(full);
                return true;
            }
            mbar_arrive_expect_tx(full, (uint32_t)NBOX * 4u);
            const int t = tile & (kCalmTile - 1);
            tma_load_3d(smem_u32(ring + b * NBOXP), &tm_in, (t % ntx) * TX - 4, (t / ntx) * TY - 3, 0, full);
            return true;
        };
        int issued = 0;
        bool ok = true;
        for (int base = 0; base < njobs && ok; base += 32) {
            const int mine = base + lane < njobs ? tiles[blockIdx.x + (base + lane) * gridDim.x] : -1;
            const int around = mine >= 0 ? fluids_around(pres_in, mine, ntx) : 0;
            const bool multi = mine >= 0 && (all || !one_fluid(around));
            for (unsigned todo = __ballot_sync(0xffffffffu, multi); todo && ok; todo &= todo - 1) {
                const int tile = __shfl_sync(0xffffffffu, around & 8 ? mine | kCalmTile : mine, __ffs(todo) - 1);
                if (lane == 0) ok = send(tile, issued);
                ok = __shfl_sync(0xffffffffu, ok, 0);
                issued += ok;
            }
        }
        if (lane != 0) return;
        // every copy issued has landed before the block may exit
        for (int m = 0; m < 2 * kRingBufs; m++) {
            int last = -1;
            for (int j = issued - 1; j >= 0 && j >= issued - 2 * kRingBufs; j--)
                if (j % (2 * kRingBufs) == m) {
                    last = j;
                    break;
                }
            if (last < 0) continue;
            const uint32_t par = (uint32_t)((last / (2 * kRingBufs)) & 1);
            for (int it = 0; it < kWaitLimit && !mbar_try_wait(smem_u32(&s_full[m]), par); it++) {
            }
        }
        if (!ok) atomicOr(P.err, 1);
        // no more tiles: one job without a copy for each group (after the waits above, which look
        // at the last copy of each barrier)
        for (int g = 0; g < 2 && ok; g++) ok = send(-1, issued + g);
        return;
    }

    // ---------------- consumer groups ----------------
    const int g = warp / NW;
    const int bar_id = 1 + g;  // named barrier of the group (0 is the block-wide one)
    const int tid = threadIdx.x - g * NT;
    const int lx = tid % TX, ly = tid / TX;
    float(*ch)[CY][CX] = s_ch[g];
    float(*rh)[CX] = s_rho[g];
    int* flags = s_flags[g];
    const bool ring_node = tid < NRING;
    int rcx = 0, rcy = 0;
    if (ring_node) {
        if (tid < 2 * CX) {
            rcx = tid % CX;
            rcy = tid / CX;
        } else if (tid < 4 * CX) {
            rcx = (tid - 2 * CX) % CX;
            rcy = CY - 2 + (tid - 2 * CX) / CX;
        } else {
            const int rr0 = tid - 4 * CX;  // 4 * TY side nodes
            const int side = rr0 / (2 * TY), rr = rr0 % (2 * TY);
            rcy = 2 + rr / 2;
            rcx = side == 0 ? (rr & 1) : CX - 2 + (rr & 1);
        }
    }
    auto store_phase = [&](int cx, int cy, float r0, float r1, float r2) {
        const float rho = (r0 + r1) + r2;
        const float ir = __fdividef(1.0f, rho);
        ch[0][cy][cx] = r0 * ir;
        ch[1][cy][cx] = r1 * ir;
        ch[2][cy][cx] = r2 * ir;
        rh[cy][cx] = rho;
        return (r0 != 0.0f ? 1 : 0) | (r1 != 0.0f ? 2 : 0) | (r2 != 0.0f ? 4 : 0);
    };

    int jj = 0;  // tiles so far that used the flags
    for (int j = g;; j += 2) {
        const float* box = ring + (j % kRingBufs) * NBOXP;
        {
            bool ok = false;
            const uint32_t full = smem_u32(&s_full[j % (2 * kRingBufs)]);
            const uint32_t par = (uint32_t)((j / (2 * kRingBufs)) & 1);
            for (int it = 0; it < P.wait_polls && !ok; it++) ok = mbar_try_wait(full, par);
            if (group_or(!ok, bar_id, NT)) {
                if (tid == 0) atomicOr(P.err, 1);
                return;
            }
        }
        const int job = s_tile[j % (2 * kRingBufs)];
        if (job < 0) return;
        const bool calm = job & kCalmTile;
        const int tile = job & (kCalmTile - 1);
        const int x0 = (tile % ntx) * TX, y0 = (tile / ntx) * TY;
        // ---- phase 1: pulls, densities and phase fields of the halo-2 region ----
        auto pull = [&](int cx, int cy, float q[27]) {
#pragma unroll
            for (int p = 0; p < kQ * kNF; p++) {
                const int a = p % kQ;
                q[p] = box[(p * BY + cy + 1 - ey(a)) * BX + cx + 2 - ex(a)];
            }
        };
        int present = 0;
        float q[27];
        if (ring_node && !calm) {
            pull(rcx, rcy, q);
            const float a0 = ((q[0] + (q[1] + q[3])) + (q[2] + q[4])) + ((q[5] + q[7]) + (q[6] + q[8]));
            const float a1 = ((q[9] + (q[10] + q[12])) + (q[11] + q[13])) + ((q[14] + q[16]) + (q[15] + q[17]));
            const float a2 = ((q[18] + (q[19] + q[21])) + (q[20] + q[22])) + ((q[23] + q[25]) + (q[24] + q[26]));
            present |= store_phase(rcx, rcy, a0, a1, a2);
        }
        float f[kQ], r0, r1, r2;
        pull(lx + 2, ly + 2, q);
        // the box is not read again: release it to the producer (all lanes of the warp are done)
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&s_empty[j % kRingBufs]));
#pragma unroll
        for (int a = 0; a < kQ; a++) f[a] = (q[a] + q[9 + a]) + q[18 + a];
        r0 = ((q[0] + (q[1] + q[3])) + (q[2] + q[4])) + ((q[5] + q[7]) + (q[6] + q[8]));
        r1 = ((q[9] + (q[10] + q[12])) + (q[11] + q[13])) + ((q[14] + q[16]) + (q[15] + q[17]));
        r2 = ((q[18] + (q[19] + q[21])) + (q[20] + q[22])) + ((q[23] + q[25]) + (q[24] + q[26]));
        if (calm) {
            // all but one fluid as traces: no gradients.  (No barrier until the next tile's, which may write
            // the phase fields: nobody reads them here.)
            const int v = collide_calm<kStoreF32>(P, Pop{fout, nullptr, nullptr}, uout, (y0 + ly) * P.nx + x0 + lx, f, r0,
                                                  r1, r2, 7);
            const int w = __reduce_or_sync(0xffffffffu, v);
            if (lane == 0) reinterpret_cast<uint8_t*>(pres_out + tile)[tid >> 5] = row_byte(w);
            continue;
        }
        present |= store_phase(lx + 2, ly + 2, r0, r1, r2);
        // fluids present in the group's phase-field region (one barrier; see fluids_present)
        int cnt;
        {
            const int w = __reduce_or_sync(0xffffffffu, present);
            if (lane == 0 && w) atomicOr(&flags[jj & 1], w);
            group_sync(bar_id, NT);
            const int v = flags[jj & 1];
            if (tid == 0) flags[(jj + 1) & 1] = 0;
            cnt = __popc(v & 7);
            jj++;
        }
        const bool mixed = cnt != 1;

        // ---- phase 2: stress tensor of Eq.(10) on the halo-1 region ----
        if (mixed) stress_halo1<TX, TY>(P, ch, rh, s_txx[g], s_txy[g], s_tyy[g], tid);
        group_sync(bar_id, NT);

        // ---- phase 3: force, collision, recolouring, 27 stores per node ----
        float Fx = 0.0f, Fy = 0.0f, gr[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
        if (mixed) {
            div_stress<RX>(s_txx[g], s_txy[g], s_tyy[g], lx + 1, ly + 1, Fx, Fy);
#pragma unroll
            for (int k = 0; k < kNF; k++) grad9_f<CX>(ch[k], lx + 2, ly + 2, gr[2 * k], gr[2 * k + 1]);
        }
        float ux, uy;
        const Recolour rc = collide_node(P, f, r0, r1, r2, Fx, Fy, gr, ux, uy);
        if (uout) {
            const int i = (y0 + ly) * P.nx + x0 + lx;
            uout[i] = ux;
            uout[P.N + i] = uy;
        }
        float* o = fout + (y0 + ly) * P.nx + x0 + lx;
#pragma unroll
        for (int k = 0; k < kNF; k++)
#pragma unroll
            for (int a = 0; a < kQ; a++)
                o[P.off_plane[k * kQ + a]] =
                    rc.C[k] * f[a] + wq(a) * (rc.Vx[k] * (float)ex(a) + rc.Vy[k] * (float)ey(a));
        // what this warp's nodes hold, for the tiles around this one in the next step
        const int w = row_bits(recoloured_bits<kStoreF32>(f, r0, r1, r2, rc), f);
        if (lane == 0) reinterpret_cast<uint8_t*>(pres_out + tile)[tid >> 5] = row_byte(w);
        // the next tile's phase fields overwrite ch / rh only after its own barriers; the stress
        // arrays after its phase-1 barrier, by which time every thread here has read them
    }
}

// ------------------------------------------------------------------------------------------
// initial state, fields, diagnostics
// ------------------------------------------------------------------------------------------
// Stored populations whose pull gives f_ak(x) = w_a rho_k(x): population a of node y is
// w_a rho_k at its destination y + e_a (or at y itself when the destination is solid).
template <int STORE>
__global__ void k_init(const Params P, const double* __restrict__ rho,
                       const uint8_t* __restrict__ type, const Pop f)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P.N) return;
    const int x = i % P.nx, y = i / P.nx;
    const bool solid = type[i] & 2;
    float v[27];
#pragma unroll
    for (int a = 0; a < kQ; a++) {
        const Loc d = locate(P, x + ex(a), y + ey(a));
#pragma unroll
        for (int k = 0; k < kNF; k++) {
            float val = 0.0f;
            if (!solid) {
                if (d.kind == 1 || (d.kind == 0 && (type[d.idx] & 2)))
                    val = wq(a) * (float)rho[(long long)k * P.N + i];
                else if (d.kind == 0)
                    val = wq(a) * (float)rho[(long long)relabel(k, d.par) * P.N + d.idx];
            }
            v[9 * k + a] = val;
        }
    }
    store_node<STORE>(f, P.N, i, v);
}

// post-streaming densities in double precision, as the caller gets them
template <class S>
__global__ void k_fields(const Params P, const S st, const uint8_t* __restrict__ type, double* __restrict__ rho_out)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P.N) return;
    float r[kNF] = {0.f, 0.f, 0.f};
    if (!(type[i] & 2)) {
        float p[27];
        pull_global(P, st, type, i % P.nx, i / P.nx, p);
#pragma unroll
        for (int k = 0; k < kNF; k++)
#pragma unroll
            for (int a = 0; a < kQ; a++) r[k] += p[9 * k + a];
    }
#pragma unroll
    for (int k = 0; k < kNF; k++) rho_out[(long long)k * P.N + i] = (double)r[k];
}

// n numbers in double precision
__global__ void k_widen(const long long n, const float* __restrict__ in, double* __restrict__ out)
{
    const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = (double)in[i];
}

// post-streaming populations of every fluid node (0 at solid nodes)
template <class S>
__global__ void k_get_state(const Params P, const S st, const uint8_t* __restrict__ type,
                            float* __restrict__ post)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P.N) return;
    float p[27];
    if (!(type[i] & 2)) {
        pull_global(P, st, type, i % P.nx, i / P.nx, p);
    } else {
#pragma unroll
        for (int j = 0; j < 27; j++) p[j] = 0.0f;
    }
#pragma unroll
    for (int j = 0; j < 27; j++) post[(long long)j * P.N + i] = p[j];
}

// stored populations whose pull reproduces the post-streaming state `post`: population a of
// node y is post_a at its destination y + e_a, or post_opp(a) at y when that destination is solid
template <int STORE>
__global__ void k_set_state(const Params P, const double* __restrict__ post,
                            const uint8_t* __restrict__ type, const Pop f)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P.N) return;
    const int x = i % P.nx, y = i / P.nx;
    const bool solid = type[i] & 2;
    float v[27];
#pragma unroll
    for (int a = 0; a < kQ; a++) {
        const Loc d = locate(P, x + ex(a), y + ey(a));
#pragma unroll
        for (int k = 0; k < kNF; k++) {
            float val = 0.0f;
            if (!solid) {
                if (d.kind == 1 || (d.kind == 0 && (type[d.idx] & 2)))
                    val = (float)post[(long long)(k * kQ + opp(a)) * P.N + i];
                else if (d.kind == 0)
                    val = (float)post[(long long)(relabel(k, d.par) * kQ + a) * P.N + d.idx];
            }
            v[9 * k + a] = val;
        }
    }
    store_node<STORE>(f, P.N, i, v);
}

constexpr int kDiagThreads = 256;

// out per block: [0..2] sum rho_k, [3] sum x rho_0, [4] sum y rho_0, [5] max|u|, [6] min rho,
// [7] non-finite count
template <class S>
__global__ void __launch_bounds__(kDiagThreads) k_diag(const Params P, const S st,
                                                       const uint8_t* __restrict__ type,
                                                       const float* __restrict__ u,
                                                       double* __restrict__ partials)
{
    double acc[8] = {0, 0, 0, 0, 0, 0, DBL_MAX, 0};
    for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < P.N;
         i += (long long)gridDim.x * blockDim.x) {
        if (type[i] & 2) continue;
        const int x = (int)(i % P.nx), y = (int)(i / P.nx);
        float p[27];
        pull_global(P, st, type, x, y, p);
        double r[kNF];
#pragma unroll
        for (int k = 0; k < kNF; k++) {
            float s = 0.f;
#pragma unroll
            for (int a = 0; a < kQ; a++) s += p[9 * k + a];
            r[k] = s;
            acc[k] += s;
            if (!isfinite(s)) acc[7] += 1.0;
        }
        acc[3] += x * r[0];
        acc[4] += y * r[0];
        const double um = sqrt((double)u[i] * u[i] + (double)u[P.N + i] * u[P.N + i]);
        acc[5] = fmax(acc[5], um);
        acc[6] = fmin(acc[6], r[0] + r[1] + r[2]);
    }
    __shared__ double sh[8][kDiagThreads];
#pragma unroll
    for (int j = 0; j < 8; j++) sh[j][threadIdx.x] = acc[j];
    __syncthreads();
    for (int s = kDiagThreads / 2; s > 0; s >>= 1) {
        if (threadIdx.x < s) {
#pragma unroll
            for (int j = 0; j < 5; j++) sh[j][threadIdx.x] += sh[j][threadIdx.x + s];
            sh[5][threadIdx.x] = fmax(sh[5][threadIdx.x], sh[5][threadIdx.x + s]);
            sh[6][threadIdx.x] = fmin(sh[6][threadIdx.x], sh[6][threadIdx.x + s]);
            sh[7][threadIdx.x] += sh[7][threadIdx.x + s];
        }
        __syncthreads();
    }
    if (threadIdx.x < 8) partials[blockIdx.x * 8 + threadIdx.x] = sh[threadIdx.x][0];
}

// one warp: lane j strides over the block partials, then a shuffle reduction
__global__ void k_diag_final(const int nb, const double* __restrict__ partials, double* __restrict__ out)
{
    double acc[8] = {0, 0, 0, 0, 0, 0, DBL_MAX, 0};
    for (int b = threadIdx.x; b < nb; b += 32) {
        const double* q = partials + 8 * b;
#pragma unroll
        for (int j = 0; j < 5; j++) acc[j] += q[j];
        acc[5] = fmax(acc[5], q[5]);
        acc[6] = fmin(acc[6], q[6]);
        acc[7] += q[7];
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
#pragma unroll
        for (int j = 0; j < 5; j++) acc[j] += __shfl_xor_sync(0xffffffffu, acc[j], o);
        acc[5] = fmax(acc[5], __shfl_xor_sync(0xffffffffu, acc[5], o));
        acc[6] = fmin(acc[6], __shfl_xor_sync(0xffffffffu, acc[6], o));
        acc[7] += __shfl_xor_sync(0xffffffffu, acc[7], o);
    }
    if (threadIdx.x == 0)
        for (int j = 0; j < 8; j++) out[j] = acc[j];
}

}  // namespace

// ------------------------------------------------------------------------------------------
// launchers
// ------------------------------------------------------------------------------------------
// call fn with the Store type of the storage format
template <class Fn>
void with_store(int store, const Pop& p, long long N, Fn fn)
{
    if (store == kStoreF32)
        fn(Store<kStoreF32>(p, N));
    else if (store == kStoreF16)
        fn(Store<kStoreF16>(p, N));
    else
        fn(Store<kStoreBF16>(p, N));
}

void launch_wet_init(int store, const Params& P, int nw, const int* widx, const Pop& f,
                     const uint8_t* type, double* Cw, cudaStream_t s)
{
    if (nw <= 0) return;
    with_store(store, f, P.N, [&](auto st) {
        k_wet_init<<<(nw + 127) / 128, 128, 0, s>>>(P, nw, widx, st, type, Cw);
    });
}

void launch_step_plain(int store, const Params& P, const int* tiles, int ntiles, const Pop& fin, const Pop& fout,
                       float* u, const uint64_t* pres_in, uint64_t* pres_out, bool all, cudaStream_t s)
{
    if (ntiles <= 0) return;
    const dim3 b(kTX, kTY);
    if (store == kStoreF32)
        k_step_plain<kTX, kTY, kStoreF32><<<ntiles, b, 0, s>>>(P, tiles, fin, fout, u, pres_in, pres_out, all);
    else if (store == kStoreF16)
        k_step_plain<kTX, kTY, kStoreF16><<<ntiles, b, 0, s>>>(P, tiles, fin, fout, u, pres_in, pres_out, all);
    else
        k_step_plain<kTX, kTY, kStoreBF16><<<ntiles, b, 0, s>>>(P, tiles, fin, fout, u, pres_in, pres_out, all);
}

cudaError_t launch_tile(int store, const Params& P, const TileSet& T, const Pop& fin, const Pop& fout, double* cw_out,
                        float* u, const uint64_t* pres_in, uint64_t* pres_out, bool full_write, bool one, bool chain,
                        cudaStream_t s)
{
    if (T.ntiles <= 0) return cudaSuccess;
    const int fw = full_write ? 1 : 0, on = one ? 1 : 0;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3(T.ntiles);
    cfg.blockDim = dim3(kTileThreads);
    cfg.stream = s;
    cfg.attrs = &attr;
    cfg.numAttrs = chain ? 1 : 0;
    auto go = [&](auto kernel) {
        return cudaLaunchKernelEx(&cfg, kernel, P, T, fin, fout, cw_out, u, pres_in, pres_out, fw, on);
    };
    if (store == kStoreF32) return go(k_tile<kTX, kTY, kStoreF32>);
    if (store == kStoreF16) return go(k_tile<kTX, kTY, kStoreF16>);
    return go(k_tile<kTX, kTY, kStoreBF16>);
}

void launch_wet_look(const Params& P, const TileSet& T, int entries, const double* Cw, cudaStream_t s)
{
    if (entries > 0) k_wet_look<<<(4 * entries + 127) / 128, 128, 0, s>>>(P, T, entries, Cw);
}

// Pure tiles of the 16-bit storage through the tensor memory accelerator, persistent, with the
// tile loop of k_step_tma: per tile one bulk copy of the FP32 densities (box (TX + 8) x (TY + 6)
// x 3 from (x0 - 4, y0 - 3)) and one of the 24 planes of 16-bit offsets (box (TX + 16) x (TY + 6)
// x 24 from (x0 - 8, y0 - 3): a 16-bit box must start on a 16-byte boundary) complete on an
// mbarrier; a pull rebuilds w_a rho_k + offset at its source, the rest population from the
// node's own offsets, exactly as the plain kernel does from global memory.  A warp's reads of
// one plane are consecutive 16-bit words (no bank conflicts).  The next tile's boxes are fetched
// as soon as the pulls are done.
template <int TX, int TY, int STORE>
__global__ void __launch_bounds__(TX* TY, kTma16BlocksPerSm) k_step_tma16(const Params P, const int* __restrict__ tiles,
                                                            const int ntiles, const Pop fout,
                                                            float* __restrict__ uout,
                                                            const __grid_constant__ CUtensorMap tm_rho,
                                                            const __grid_constant__ CUtensorMap tm_off,
                                                            const uint64_t* __restrict__ pres_in,
                                                            uint64_t* __restrict__ pres_out, const int all)
{
    constexpr int NT = TX * TY;
    constexpr int CX = TX + 4, CY = TY + 4;
    constexpr int RX = TX + 2, RY = TY + 2;
    constexpr int BX = TX + 8, BY = TY + 6;          // density box
    constexpr int OX = TX + 16;                      // width of the offset box
    constexpr int NR = kNF * BY * BX;                // floats of the density box
    constexpr int NRP = (NR + 31) / 32 * 32;         // keeps the offset box 128-byte aligned
    constexpr int PO = BY * OX;                      // 16-bit words of one offset plane
    constexpr uint32_t kBytes = NR * 4u + 24u * PO * 2u;  // both copies
    __shared__ float s_ch[kNF][CY][CX];
    __shared__ float s_rho[CY][CX];
    __shared__ float s_txx[RY][RX], s_txy[RY][RX], s_tyy[RY][RX];
    __shared__ __align__(8) uint64_t s_bar;
    __shared__ int s_flags[2];   // fluids present in the tile, by iteration parity
    __shared__ int s_list[NT];   // tiles of the current batch
    __shared__ int s_wn[NT / 32];
    extern __shared__ unsigned char dsm[];
    float* rbox = reinterpret_cast<float*>(dsm + ((128u - (smem_u32(dsm) & 127u)) & 127u));  // [3][BY][BX]
    const unsigned short* obox = reinterpret_cast<const unsigned short*>(rbox + NRP);          // [24][BY][OX]

    const int tid = threadIdx.x + TX * threadIdx.y;
    const int lx = threadIdx.x, ly = threadIdx.y;
    const int ntx = (P.nx + TX - 1) / TX;
    const uint32_t bar = smem_u32(&s_bar);
    if ((int)blockIdx.x >= ntiles) return;
    auto issue = [&](int tile) {
        const int x0 = (tile % ntx) * TX, y0 = (tile / ntx) * TY;
        mbar_arrive_expect_tx(bar, kBytes);
        tma_load_3d(smem_u32(rbox), &tm_rho, x0 - 4, y0 - 3, 0, bar);
        tma_load_3d(smem_u32(obox), &tm_off, x0 - 8, y0 - 3, 0, bar);
    };
    int last = -1;
    if (tid == 0) {
        mbar_init(bar, 1);
        fence_mbar_init();
        s_flags[0] = s_flags[1] = 0;
    }

    // pull of the node at (cx, cy) of the phase-field region from the boxes
    auto pull = [&](int cx, int cy, float q[27]) {
        const int own = (cy + 1) * BX + cx + 2, owno = (cy + 1) * OX + cx + 6;
#pragma unroll
        for (int k = 0; k < kNF; k++) {
            const float rk = rbox[k * BY * BX + own];
            float d[kQ];
#pragma unroll
            for (int a = 1; a < kQ; a++) d[a] = dec16<STORE>(obox[(8 * k + a - 1) * PO + owno]);
            q[9 * k] = wq(0) * rk - sum_offsets(d);
#pragma unroll
            for (int a = 1; a < kQ; a++) {
                const int src = k * BY * BX + (cy + 1 - ey(a)) * BX + cx + 2 - ex(a);
                const int srco = (8 * k + a - 1) * PO + (cy + 1 - ey(a)) * OX + cx + 6 - ex(a);
                q[9 * k + a] = wq(a) * rbox[src] + dec16<STORE>(obox[srco]);
            }
        }
    };
    auto store_phase = [&](int cx, int cy, const float q[27]) {
        float r[kNF];
#pragma unroll
        for (int k = 0; k < kNF; k++) {
            const float* qk = q + 9 * k;
            r[k] = ((qk[0] + (qk[1] + qk[3])) + (qk[2] + qk[4])) + ((qk[5] + qk[7]) + (qk[6] + qk[8]));
        }
        const float rho = (r[0] + r[1]) + r[2];
        const float ir = __fdividef(1.0f, rho);
#pragma unroll
        for (int k = 0; k < kNF; k++) s_ch[k][cy][cx] = r[k] * ir;
        s_rho[cy][cx] = rho;
        return (r[0] != 0.0f ? 1 : 0) | (r[1] != 0.0f ? 2 : 0) | (r[2] != 0.0f ? 4 : 0);
    };

    int j = 0;
    const int mine = (ntiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
    // the block's tiles in batches of one candidate per thread: those with one fluid around are
    // k_step_one's, the others are listed
    for (int base = 0; base < mine; base += NT) {
        const int cand = base + tid < mine ? tiles[blockIdx.x + (base + tid) * gridDim.x] : -1;
        const int around = cand >= 0 ? fluids_around(pres_in, cand, ntx) : 0;
        const bool multi = cand >= 0 && (all || !one_fluid(around));
        const unsigned votes = __ballot_sync(0xffffffffu, multi);
        if ((tid & 31) == 0) s_wn[tid >> 5] = __popc(votes);
        __syncthreads();  // the counts, and every thread is past the last batch's list
        int pos = __popc(votes & ((1u << (tid & 31)) - 1)), count = 0;
        for (int w = 0; w < NT / 32; w++) {
            if (w < (tid >> 5)) pos += s_wn[w];
            count += s_wn[w];
        }
        if (multi) s_list[pos] = around & 8 ? cand | kCalmTile : cand;
        __syncthreads();
        if (tid == 0 && count > 0) {
            issue(s_list[0] & (kCalmTile - 1));
            last = j;
        }
        for (int m = 0; m < count; m++, j++) {
            const bool more = m + 1 < count;
            const bool calm = s_list[m] & kCalmTile;
            const int tile = s_list[m] & (kCalmTile - 1);
            const int x0 = (tile % ntx) * TX, y0 = (tile / ntx) * TY;
            bool ok = false;
            for (int it = 0; it < P.wait_polls && !ok; it++) ok = mbar_try_wait(bar, j & 1);
            if (__syncthreads_or(!ok)) {
                // the copies did not complete in time: record it, give them a second bounded wait
                // so that they do not land in a later block's shared memory, and stop
                if (tid == 0) {
                    atomicOr(P.err, 1);
                    for (int it = 0; last >= 0 && it < kWaitLimit && !mbar_try_wait(bar, last & 1); it++) {
                    }
                }
                return;
            }

            // ---- phase 1: pulls, densities and phase fields of the halo-2 region ----
            int present = 0;
            {
                constexpr int NRING = CX * CY - TX * TY;
                for (int r = tid; r < NRING && !calm; r += NT) {
                    int cx, cy;
                    if (r < 2 * CX) {
                        cx = r % CX;
                        cy = r / CX;
                    } else if (r < 4 * CX) {
                        cx = (r - 2 * CX) % CX;
                        cy = CY - 2 + (r - 2 * CX) / CX;
                    } else {
                        const int rr0 = r - 4 * CX;  // 4 * TY side nodes
                        const int side = rr0 / (2 * TY), rr = rr0 % (2 * TY);
                        cy = 2 + rr / 2;
                        cx = side == 0 ? (rr & 1) : CX - 2 + (rr & 1);
                    }
                    float q[27];
                    pull(cx, cy, q);
                    present |= store_phase(cx, cy, q);
                }
            }
            float f[kQ], r0, r1, r2;
            {
                float q[27];
                pull(lx + 2, ly + 2, q);
                if (!calm) present |= store_phase(lx + 2, ly + 2, q);
#pragma unroll
                for (int a = 0; a < kQ; a++) f[a] = (q[a] + q[9 + a]) + q[18 + a];
                r0 = ((q[0] + (q[1] + q[3])) + (q[2] + q[4])) + ((q[5] + q[7]) + (q[6] + q[8]));
                r1 = ((q[9] + (q[10] + q[12])) + (q[11] + q[13])) + ((q[14] + q[16]) + (q[15] + q[17]));
                r2 = ((q[18] + (q[19] + q[21])) + (q[20] + q[22])) + ((q[23] + q[25]) + (q[24] + q[26]));
            }
            const bool mixed = fluids_present(present, s_flags, j, tid) != 1;
            // the boxes are free: fetch the next tile's while this one computes
            if (tid == 0 && more) {
                issue(s_list[m + 1] & (kCalmTile - 1));
                last = j + 1;
            }

            const int i = (y0 + ly) * P.nx + x0 + lx;
            if (calm) {
                // all but one fluid as traces: no gradients
                const int w = __reduce_or_sync(0xffffffffu, collide_calm<STORE>(P, fout, uout, i, f, r0, r1, r2, 7));
                if ((tid & 31) == 0) reinterpret_cast<uint8_t*>(pres_out + tile)[tid >> 5] = row_byte(w);
                continue;
            }

            // ---- phase 2: stress tensor of Eq.(10) on the halo-1 region ----
            if (mixed) stress_halo1<TX, TY>(P, s_ch, s_rho, s_txx, s_txy, s_tyy, tid);
            __syncthreads();

            // ---- phase 3: force, collision, recolouring, 16-bit stores ----
            float Fx = 0.0f, Fy = 0.0f, g[6] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
            if (mixed) {
                div_stress<RX>(s_txx, s_txy, s_tyy, lx + 1, ly + 1, Fx, Fy);
#pragma unroll
                for (int k = 0; k < kNF; k++) grad9_f<CX>(s_ch[k], lx + 2, ly + 2, g[2 * k], g[2 * k + 1]);
            }
            float ux, uy;
            const Recolour rc = collide_node(P, f, r0, r1, r2, Fx, Fy, g, ux, uy);
            if (uout) {
                uout[i] = ux;
                uout[P.N + i] = uy;
            }
            float v[27];
#pragma unroll
            for (int k = 0; k < kNF; k++)
#pragma unroll
                for (int a = 0; a < kQ; a++)
                    v[9 * k + a] = rc.C[k] * f[a] + wq(a) * (rc.Vx[k] * (float)ex(a) + rc.Vy[k] * (float)ey(a));
            store_node<STORE>(fout, P.N, i, v);
            // what this warp's nodes hold, for the tiles around this one in the next step
            const int w = row_bits(recoloured_bits<STORE>(f, r0, r1, r2, rc), f);
            if ((tid & 31) == 0) reinterpret_cast<uint8_t*>(pres_out + tile)[tid >> 5] = row_byte(w);
        }
    }
}

// output path of the TMA kernel: staged in shared memory and written by one bulk tensor store per
// tile, or written directly (a smaller shared-memory footprint leaves room on each SM for blocks
// of the wall-tile kernel, which runs concurrently)
constexpr bool kTmaStage = false;

size_t step_tma_smem_bytes()
{
    const size_t nbox = ((size_t)kQ * kNF * (kTY + 6) * (kTX + 8) + 31) / 32 * 32;
    return (nbox + (kTmaStage ? (size_t)kQ * kNF * kTY * kTX : 0)) * sizeof(float) + 128u;
}

cudaError_t step_tma_prepare()
{
    return cudaFuncSetAttribute(k_step_tma<kTX, kTY, kTmaStage>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)step_tma_smem_bytes());
}

void launch_step_tma(const Params& P, const int* tiles, int ntiles, int nblocks, const Pop& fout, float* u,
                     const CUtensorMap& tin_a, const CUtensorMap& tin_b, const CUtensorMap& tout, uint64_t* pres_out,
                     cudaStream_t s)
{
    if (ntiles <= 0) return;
    const int nb = nblocks < ntiles ? nblocks : ntiles;
    k_step_tma<kTX, kTY, kTmaStage>
        <<<nb, dim3(kTX, kTY), step_tma_smem_bytes(), s>>>(P, tiles, ntiles, fout.f, u, tin_a, tin_b, tout, pres_out);
}

size_t step_ring_smem_bytes()
{
    const size_t nbox = ((size_t)kQ * kNF * (kTY + 6) * (kTX + 8) + 31) / 32 * 32;
    return (size_t)kRingBufs * nbox * sizeof(float) + 128u;
}

cudaError_t step_ring_prepare()
{
    return cudaFuncSetAttribute(k_step_ring<kTX, kTY>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                (int)step_ring_smem_bytes());
}

void launch_step_ring(const Params& P, const int* tiles, int ntiles, int nblocks, const Pop& fout, float* u,
                      const CUtensorMap& tin, const uint64_t* pres_in, uint64_t* pres_out, bool all, cudaStream_t s)
{
    if (ntiles <= 0) return;
    const int nb = nblocks < ntiles ? nblocks : ntiles;
    k_step_ring<kTX, kTY><<<nb, 2 * kTX * kTY + 32, step_ring_smem_bytes(), s>>>(P, tiles, ntiles, fout.f, u, tin,
                                                                                 pres_in, pres_out, all);
}

size_t step_tma16_smem_bytes()
{
    const size_t nr = ((size_t)kNF * (kTY + 6) * (kTX + 8) + 31) / 32 * 32;
    return nr * sizeof(float) + (size_t)24 * (kTY + 6) * (kTX + 16) * sizeof(unsigned short) + 128u;
}

// the 16-bit offset box takes the block past the 48 KB of shared memory a kernel gets without
// opting in
cudaError_t step_tma16_prepare()
{
    cudaError_t e = cudaFuncSetAttribute(k_step_tma16<kTX, kTY, kStoreF16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                         (int)step_tma16_smem_bytes());
    if (e == cudaSuccess)
        e = cudaFuncSetAttribute(k_step_tma16<kTX, kTY, kStoreBF16>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 (int)step_tma16_smem_bytes());
    return e;
}

void launch_step_tma16(int store, const Params& P, const int* tiles, int ntiles, int nblocks, const Pop& fout,
                       float* u, const CUtensorMap& trho, const CUtensorMap& toff, const uint64_t* pres_in,
                       uint64_t* pres_out, bool all, cudaStream_t s)
{
    if (ntiles <= 0) return;
    const int nb = nblocks < ntiles ? nblocks : ntiles;
    if (store == kStoreF16)
        k_step_tma16<kTX, kTY, kStoreF16><<<nb, dim3(kTX, kTY), step_tma16_smem_bytes(), s>>>(
            P, tiles, ntiles, fout, u, trho, toff, pres_in, pres_out, all);
    else
        k_step_tma16<kTX, kTY, kStoreBF16><<<nb, dim3(kTX, kTY), step_tma16_smem_bytes(), s>>>(
            P, tiles, ntiles, fout, u, trho, toff, pres_in, pres_out, all);
}

void launch_count(const Params& P, const int* tiles, int ntiles, const uint64_t* pres, unsigned* out, cudaStream_t s)
{
    if (ntiles > 0) k_count<<<(ntiles + 255) / 256, 256, 0, s>>>(P, tiles, ntiles, pres, out);
}

void launch_step_one(int store, const Params& P, const TileSet& T, const int* tiles, int ntiles, const Pop& fin,
                     const Pop& fout, float* u, const uint64_t* pres_in, uint64_t* pres_out, bool full_write,
                     cudaStream_t s)
{
    constexpr int per = kOneThreads / 32;
    const int fw = full_write ? 1 : 0;
    const unsigned nb = (unsigned)(((long long)ntiles * (kTY / kOneRows) + per - 1) / per);
    const unsigned ng = (unsigned)(((long long)T.ntiles * kTY + per - 1) / per);
    auto go = [&](auto pure, auto general) {
        if (nb > 0) pure<<<nb, kOneThreads, 0, s>>>(P, T, tiles, ntiles, fin, fout, u, pres_in, pres_out, fw);
        if (ng > 0) general<<<ng, kOneThreads, 0, s>>>(P, T, tiles, ntiles, fin, fout, u, pres_in, pres_out, fw);
    };
    if (store == kStoreF32)
        go(k_step_one<kTX, kTY, kStoreF32, true>, k_step_one<kTX, kTY, kStoreF32, false>);
    else if (store == kStoreF16)
        go(k_step_one<kTX, kTY, kStoreF16, true>, k_step_one<kTX, kTY, kStoreF16, false>);
    else
        go(k_step_one<kTX, kTY, kStoreBF16, true>, k_step_one<kTX, kTY, kStoreBF16, false>);
}

void launch_init(int store, const Params& P, const double* rho, const uint8_t* type, const Pop& f,
                 cudaStream_t s)
{
    const unsigned nb = (unsigned)((P.N + 255) / 256);
    if (store == kStoreF32)
        k_init<kStoreF32><<<nb, 256, 0, s>>>(P, rho, type, f);
    else if (store == kStoreF16)
        k_init<kStoreF16><<<nb, 256, 0, s>>>(P, rho, type, f);
    else
        k_init<kStoreBF16><<<nb, 256, 0, s>>>(P, rho, type, f);
}

void launch_fields(int store, const Params& P, const Pop& f, const uint8_t* type, double* rho_out, cudaStream_t s)
{
    with_store(store, f, P.N, [&](auto st) {
        k_fields<<<(unsigned)((P.N + 255) / 256), 256, 0, s>>>(P, st, type, rho_out);
    });
}

void launch_widen(long long n, const float* in, double* out, cudaStream_t s)
{
    k_widen<<<(unsigned)((n + 255) / 256), 256, 0, s>>>(n, in, out);
}

void launch_get_state(int store, const Params& P, const Pop& f, const uint8_t* type, float* post,
                      cudaStream_t s)
{
    with_store(store, f, P.N, [&](auto st) {
        k_get_state<<<(unsigned)((P.N + 255) / 256), 256, 0, s>>>(P, st, type, post);
    });
}

void launch_set_state(int store, const Params& P, const double* post, const uint8_t* type,
                      const Pop& f, cudaStream_t s)
{
    const unsigned nb = (unsigned)((P.N + 255) / 256);
    if (store == kStoreF32)
        k_set_state<kStoreF32><<<nb, 256, 0, s>>>(P, post, type, f);
    else if (store == kStoreF16)
        k_set_state<kStoreF16><<<nb, 256, 0, s>>>(P, post, type, f);
    else
        k_set_state<kStoreBF16><<<nb, 256, 0, s>>>(P, post, type, f);
}

int diag_blocks(const Params& P)
{
    long long b = (P.N + kDiagThreads - 1) / kDiagThreads;
    return (int)(b < 1216 ? b : 1216);
}

void launch_diag(int store, const Params& P, const Pop& f, const uint8_t* type, const float* u,
                 double* partials, double* out, cudaStream_t s)
{
    const int nb = diag_blocks(P);
    with_store(store, f, P.N, [&](auto st) {
        k_diag<<<nb, kDiagThreads, 0, s>>>(P, st, type, u, partials);
    });
    k_diag_final<<<1, 32, 0, s>>>(nb, partials, out);
}

}  // namespace lbm3k
