// Differentiation of the switching work W(theta) = sum_k dH/dlambda(x_k) (lambda_{k+1} - lambda_k)
// (Eq. Wdyn, left point) with respect to the SW parameters theta = (A, B, p, q, a, lambda3,
// gamma), through the Langevin velocity-Verlet trajectory with the thermostat noise held fixed.
//
// Building block: one FP64 kernel evaluates the SW energy, forces and dU/dtheta in dual numbers
// v + eps d, the dual direction being a displacement w of every atom together with a parameter
// direction dtheta.  The dual parts are then
//   F'  = J w + (dF/dtheta) dtheta          (J = dF/dx = -Hessian, symmetric)
//   E'  = -F . w + (dU/dtheta) . dtheta
//   G'  = (d2U/dtheta dx) w + (d2U/dtheta2) dtheta    (G = dU/dtheta)
// which are the Hessian-vector and mixed products that both the tangent-linear run and the
// reverse (adjoint) sweep need.  Every sum runs in a fixed order, so every output is reproducible
// bit for bit.
//
// The adjoint context integrates its own FP64 NVT trajectory (Frenkel-Ladd or reversible
// scaling, same update as the engine's FP64 path), keeps (x, v, F) every K_c steps, and in the
// reverse sweep recomputes each segment from its checkpoint before stepping the adjoint
// variables back through it.
#include <cstddef>
#include <cstdint>
#include <cstring>
#include <vector>

#include "nefe.h"
#include "nefe_dev.h"
#include "nefe_host.h"
#include "nefe_launch.h"
#include "nefe_nvtx.h"
#include "nefe_sw_terms.h"

namespace nefe {
namespace ad {

constexpr int kAdThreads = 128;
constexpr int kRed = 16;     // [E, E', G(7), G'(7)]

// ------------------------------------------------------------------------------------
// SW evaluation: k_sw_edges (shells, edge terms, leg forces), k_sw_gather (forces).
//
// Both are bound by FP64 issue (2 lanes a cycle and SM, so a warp instruction occupies the unit
// for 16 cycles whatever its active lanes).  What that asks for:
//   * the Verlet row is filtered in FP32 on fixed-point fractional positions, so FP64 sees only
//     the edges (10.6 of 18.8 entries in the liquid);
//   * the edges of a warp's atoms form one list that its lanes walk 32 at a time, so no lane
//     idles while another atom has more edges;
//   * each triplet force is computed once, through the shell's moments, stored per edge and read
//     by the leg atom's gather, where the plain form recomputed every neighbour's shell.
// 32,768-atom liquid: 3593 -> 149 us (plain), 7669 -> 376 us (dual numbers, with dU/dtheta).
// ------------------------------------------------------------------------------------
constexpr int kAdShell = 32;      // edges inside the cutoff an atom may have
constexpr int kAdCand = 40;       // candidates (FP32 filter with its margin)
constexpr int kAdEdges = 512;     // edges of one batch of a warp
constexpr int kAdComp = 7;        // values kept per edge between its phases
constexpr int kAdMaxWarps = 152 * 16;

template <typename T, typename TP>
struct AdArgs {
    const double* x;     // SoA [3n]
    const double* w;     // SoA [3n] dual direction of x (NULL: zero)
    int n, apw;          // atoms, atoms per warp (8, 16 or 32)
    double L[3], iL[3];
    float Lf[3];         // L 2^-32
    float rcf2;          // cutoff squared with the filter's margin
    const int4* xf;      // fractional positions
    int4* xf_ref;        // their values at the last list build, refreshed when *rebuild (or NULL)
    const int* rebuild;
    const int* nbr;
    const int* cnt;
    int cap, row4;       // row4: rows can be read 16 bytes at a time
    SWp<TP> P;
    int* shj;            // [n][kAdCand] candidate neighbours
    int* shn;            // [n]
    T* eb;               // [warps][kAdComp][kAdEdges]
    T* leg;              // [n][kAdCand][3] force on the leg atom of each edge
    double* part;        // [warps][kRed] partial sums
    unsigned* err;
};

template <typename T, typename TP>
__device__ __forceinline__ void edge_vector(const AdArgs<T, TP>& A, int i, int j, double (&d)[3], double (&w)[3]) {
    const size_t N = (size_t)A.n;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const double raw = __dsub_rn(A.x[k * N + j], A.x[k * N + i]);
        d[k] = __fma_rn(-A.L[k], rint(__dmul_rn(raw, A.iL[k])), raw);
        w[k] = 0.0;
        if constexpr (is_dual<T>::value)
            if (A.w) w[k] = __dsub_rn(A.w[k * N + j], A.w[k * N + i]);
    }
}

// Edges inside the cutoff of atom i (only where its candidates exceed kAdShell).
template <typename T, typename TP>
__device__ __noinline__ int count_shell(const AdArgs<T, TP>& A, int i, int m) {
    int c = 0;
    for (int a = 0; a < m; ++a) {
        double d[3], w[3];
        edge_vector(A, i, A.shj[(size_t)i * kAdCand + a], d, w);
        const double r2 = __fma_rn(d[2], d[2], __fma_rn(d[1], d[1], __dmul_rn(d[0], d[0])));
        c += r2 < A.P.rc2 ? 1 : 0;
    }
    return c;
}

// One warp per block; each warp takes groups of apw consecutive atoms.
template <typename T, typename TP, bool GRAD>
__global__ void __launch_bounds__(32) k_sw_edges(const __grid_constant__ AdArgs<T, TP> A) {
    constexpr unsigned kAll = 0xffffffffu;
    __shared__ unsigned short map[kAdEdges];     // edge -> slot << 5 | atom of the group
    __shared__ T mom[10][32];
    const SWp<TP>& P = A.P;
    const int lane = threadIdx.x;
    const unsigned below = (1u << lane) - 1u;
    T* eb = A.eb + (size_t)blockIdx.x * kAdComp * kAdEdges;
    T en = T{}, pg[7] = {};
    const int groups = (A.n + A.apw - 1) / A.apw;
    for (int g = blockIdx.x; g < groups; g += gridDim.x) {
        const int i0 = g * A.apw, i = i0 + lane;
        const bool valid = lane < A.apw && i < A.n;
        int m = 0;
        if (valid) {
            const int4 xi = A.xf[i];
            if (A.xf_ref && *A.rebuild) A.xf_ref[i] = xi;
            const int ci = min(A.cnt[i], A.cap);
            const int* row = A.nbr + (size_t)i * A.cap;
            int* sj = A.shj + (size_t)i * kAdCand;
            for (int b0 = 0; b0 < ci; b0 += 4) {
                int j[4];
                if (A.row4) {
                    const int4 r = *reinterpret_cast<const int4*>(row + b0);
                    j[0] = r.x; j[1] = r.y; j[2] = r.z; j[3] = r.w;
                } else {
#pragma unroll
                    for (int u = 0; u < 4; ++u) j[u] = b0 + u < ci ? row[b0 + u] : 0;
                }
                int4 xj[4];
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    j[u] &= (int)kIndexMask;
                    if (b0 + u < ci) xj[u] = A.xf[j[u]];
                }
#pragma unroll
                for (int u = 0; u < 4; ++u) {
                    if (b0 + u >= ci) continue;
                    const float dx = (float)wrap_sub(xj[u].x, xi.x) * A.Lf[0], dy = (float)wrap_sub(xj[u].y, xi.y) * A.Lf[1],
                                dz = (float)wrap_sub(xj[u].z, xi.z) * A.Lf[2];
                    if (dx * dx + dy * dy + dz * dz < A.rcf2) {
                        if (m < kAdCand) sj[m] = j[u];
                        ++m;
                    }
                }
            }
            if (m > kAdShell && (m > kAdCand || count_shell(A, i, m) > kAdShell))
                atomicOr(A.err, NEFE_ERR_SHELL_OVERFLOW);
            m = min(m, kAdCand);
            A.shn[i] = m;
        }
        __syncwarp();
        int incl = m;                            // edges of atoms 0 .. lane of the group
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(kAll, incl, o);
            if (lane >= o) incl += y;
        }
        int done = 0;                            // edges of the batches so far
        const int total = __shfl_sync(kAll, incl, 31);
        while (done < total) {
            // the batch: the next atoms whose edges fit kAdEdges together (at least 12 atoms)
            const bool act = incl - m >= done && incl - done <= kAdEdges && m > 0;
            const int mx = __reduce_max_sync(kAll, act ? m : 0);
            int E = 0;
            for (int a = 0; a < mx; ++a) {       // slot by slot: lanes on consecutive edges, distinct atoms
                const unsigned bal = __ballot_sync(kAll, act && a < m);
                if (act && a < m) map[E + __popc(bal & below)] = (unsigned short)(a << 5 | lane);
                E += __popc(bal);
            }
            __syncwarp();
            for (int e = lane; e < E; e += 32) { // edge terms
                const int ai = i0 + (map[e] & 31), a = map[e] >> 5;
                double d[3], w[3];
                edge_vector(A, ai, A.shj[(size_t)ai * kAdCand + a], d, w);
                EdgeT<T> t;
                sw_edge_terms<T, TP, GRAD>(P, d, w, t);
                en = fma_(0.5, t.phi, en);
                if constexpr (GRAD)
                    for (int k = 0; k < 5; ++k) pg[k] = fma_(0.5, t.pg[k], pg[k]);
                eb[0 * kAdEdges + e] = t.ux; eb[1 * kAdEdges + e] = t.uy; eb[2 * kAdEdges + e] = t.uz;
                eb[3 * kAdEdges + e] = t.g;  eb[4 * kAdEdges + e] = t.ir; eb[5 * kAdEdges + e] = t.id;
                eb[6 * kAdEdges + e] = t.dphi;
            }
            __syncwarp();
            MomT<T> M = {};
            int base = 0;
            for (int a = 0; a < mx; ++a) {       // moments, one atom per lane
                const unsigned bal = __ballot_sync(kAll, act && a < m);
                if (act && a < m) {
                    const int e = base + __popc(bal & below);
                    mom_add(M, eb[e], eb[kAdEdges + e], eb[2 * kAdEdges + e], eb[3 * kAdEdges + e]);
                }
                base += __popc(bal);
            }
            mom[0][lane] = M.G;  mom[1][lane] = M.x;  mom[2][lane] = M.y;  mom[3][lane] = M.z;
            mom[4][lane] = M.xx; mom[5][lane] = M.yy; mom[6][lane] = M.zz;
            mom[7][lane] = M.xy; mom[8][lane] = M.xz; mom[9][lane] = M.yz;
            __syncwarp();
            for (int e = lane; e < E; e += 32) { // leg forces
                const int t = map[e] & 31, a = map[e] >> 5;
                MomT<T> Q;
                Q.G = mom[0][t];  Q.x = mom[1][t];  Q.y = mom[2][t];  Q.z = mom[3][t];
                Q.xx = mom[4][t]; Q.yy = mom[5][t]; Q.zz = mom[6][t];
                Q.xy = mom[7][t]; Q.xz = mom[8][t]; Q.yz = mom[9][t];
                const T gg = eb[3 * kAdEdges + e], id = eb[5 * kAdEdges + e];
                T lx, ly, lz, s3;
                sw_leg(P, Q, eb[e], eb[kAdEdges + e], eb[2 * kAdEdges + e], eb[4 * kAdEdges + e], id, gg,
                       eb[6 * kAdEdges + e], lx, ly, lz, s3);
                T* out = A.leg + ((size_t)(i0 + t) * kAdCand + a) * 3;
                out[0] = lx; out[1] = ly; out[2] = lz;
                const T gs = mul_(gg, s3);                       // g_a S3: sum over b of g_a g_b (c - c0)^2
                const T h = mul_(mul_(P.eps, P.lam), gs);        // the triplets of edge a (each seen from both its edges)
                en = fma_(0.5, h, en);
                if constexpr (GRAD) {
                    const T hi = mul_(h, id);
                    pg[4] = fma_(mul_(P.gam, hi), id, pg[4]);
                    pg[5] = fma_(0.5 * P.eps, gs, pg[5]);
                    pg[6] = pg[6] + hi;
                }
            }
            done = __reduce_max_sync(kAll, act ? incl : 0);
            __syncwarp();
        }
    }
    double red[kRed] = {val(en), dua(en), val(pg[0]), val(pg[1]), val(pg[2]), val(pg[3]), val(pg[4]), val(pg[5]), val(pg[6]),
                        dua(pg[0]), dua(pg[1]), dua(pg[2]), dua(pg[3]), dua(pg[4]), dua(pg[5]), dua(pg[6])};
    if (!isfinite(red[0])) atomicOr(A.err, NEFE_ERR_NAN);
#pragma unroll
    for (int k = 0; k < kRed; ++k) {
        const bool used = k == 0 || (k == 1 && is_dual<T>::value) || (k >= 2 && k < 9 && GRAD) ||
                          (k >= 9 && GRAD && is_dual<T>::value);
        if (used) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) red[k] += __shfl_xor_sync(kAll, red[k], o);
        }
        if (lane == 0) A.part[(size_t)blockIdx.x * kRed + k] = red[k];
    }
}

// Force on each atom, 4 lanes per atom: minus its own edges' leg forces plus the leg forces its
// neighbours' edges exert on it (found by its index in the neighbour's shell; shells are symmetric
// because the filter distance of (i, j) and (j, i) is the same number).
template <typename T>
__global__ void __launch_bounds__(kAdThreads) k_sw_gather(int n, const int* shj, const int* shn, const T* leg, double* f,
                                                          double* fd, unsigned* err, int* rebuild) {
    if (rebuild && blockIdx.x == 0 && threadIdx.x == 0) *rebuild = 0;   // the lists are built
    const int i = (blockIdx.x * kAdThreads + threadIdx.x) >> 2, lane = threadIdx.x & 3;
    T s[3] = {};
    if (i < n) {
        const int m = shn[i];
        for (int a = lane; a < m; a += 4) {
            const int j = shj[(size_t)i * kAdCand + a];
            const T* own = leg + ((size_t)i * kAdCand + a) * 3;
            const int mj = shn[j];
            const int4* row = reinterpret_cast<const int4*>(shj + (size_t)j * kAdCand);
            int pos = -1;
            for (int b = 0; b < mj && pos < 0; b += 4) {
                const int4 r = row[b >> 2];
                pos = r.x == i ? b : (r.y == i && b + 1 < mj) ? b + 1 : (r.z == i && b + 2 < mj) ? b + 2
                      : (r.w == i && b + 3 < mj) ? b + 3 : -1;
            }
            const T* far = leg + ((size_t)j * kAdCand + (pos < 0 ? 0 : pos)) * 3;
#pragma unroll
            for (int k = 0; k < 3; ++k) s[k] = s[k] + (pos < 0 ? -own[k] : far[k] - own[k]);
        }
    }
#pragma unroll
    for (int o = 2; o > 0; o >>= 1)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            if constexpr (is_dual<T>::value)
                s[k] = s[k] + mk(__shfl_xor_sync(0xffffffffu, s[k].v, o), __shfl_xor_sync(0xffffffffu, s[k].d, o));
            else
                s[k] = s[k] + __shfl_xor_sync(0xffffffffu, s[k], o);
        }
    if (i < n && lane < 3) {
        const T v = lane == 0 ? s[0] : lane == 1 ? s[1] : s[2];
        f[(size_t)lane * n + i] = val(v);
        if (fd) fd[(size_t)lane * n + i] = dua(v);
        if (!isfinite(val(v))) atomicOr(err, NEFE_ERR_NAN);
    }
}

// Fractional positions; with ref, also whether some atom is further than the list allows from
// where the lists were built (thr2: squared displacement; always when force is set).
struct FracArgs {
    double iL[3];
    float Lf[3], thr2;
    int force;
};
__device__ __forceinline__ void frac_atom(const FracArgs& F, int i, const double (&x)[3], int4* xf, const int4* ref,
                                          int* rebuild) {
    const int4 f = make_int4(frac32(x[0], F.iL[0]), frac32(x[1], F.iL[1]), frac32(x[2], F.iL[2]), 0);
    xf[i] = f;
    if (!ref) return;
    const int4 r = ref[i];
    const float dx = (float)wrap_sub(f.x, r.x) * F.Lf[0], dy = (float)wrap_sub(f.y, r.y) * F.Lf[1],
                dz = (float)wrap_sub(f.z, r.z) * F.Lf[2];
    if (F.force || !(dx * dx + dy * dy + dz * dz < F.thr2)) *rebuild = 1;
}
__global__ void __launch_bounds__(kAdThreads) k_frac(int n, FracArgs F, const double* x, int4* xf, const int4* ref,
                                                     int* rebuild) {
    const int i = blockIdx.x * kAdThreads + threadIdx.x;
    if (i >= n) return;
    const size_t N = (size_t)n;
    const double xx[3] = {x[i], x[N + i], x[2 * N + i]};
    frac_atom(F, i, xx, xf, ref, rebuild);
}

// One warp per column; used by the noise and spring sums.
__device__ __forceinline__ void warp_block_sum(double (&v)[kRed], int used, double* out_block) {
    __shared__ double red[kAdThreads / 32][kRed];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < kRed; ++k) {
        if (k >= used) break;
        double x = v[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) red[w][k] = x;
    }
    __syncthreads();
    if (threadIdx.x < kRed) {
        double s = 0.0;
        if ((int)threadIdx.x < used)
            for (int i = 0; i < kAdThreads / 32; ++i) s += red[i][threadIdx.x];
        out_block[threadIdx.x] = s;
    }
}

// Column sums of nb rows of kRed values, each in a fixed order, one block per column (and, for
// blocks from kRed on, of a second table).
__global__ void __launch_bounds__(128) k_sum_rows(const double* part, int nb, double* out, const double* part2, int nb2,
                                                  double* out2) {
    __shared__ double red[4];
    int c = blockIdx.x;
    if (c >= kRed) {
        c -= kRed;
        part = part2; nb = nb2; out = out2;
    }
    double s = 0.0;
    for (int b = threadIdx.x; b < nb; b += 128) s += part[(size_t)b * kRed + c];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) out[c] = ((red[0] + red[1]) + red[2]) + red[3];
}

inline int ad_blocks(int n) { return (n + kAdThreads - 1) / kAdThreads; }

// Atoms per warp: 32 keeps every lane busy in the per-atom phases; fewer give small systems more
// warps (700 atoms: 22 -> 88).  The line lies where 16 (8) atoms still give about 13 (6.7) warps a SM.
inline int atoms_per_warp(int n) { return n > 48 * 1024 ? 32 : n > 8 * 1024 ? 16 : 8; }
inline int ad_warps(int n) {
    const int g = (n + atoms_per_warp(n) - 1) / atoms_per_warp(n);
    return g < kAdMaxWarps ? (g > 0 ? g : 1) : kAdMaxWarps;
}

// Scratch of an evaluation, sized for dual numbers.
struct EvalBufs {
    int4* xf = nullptr;
    int *shj = nullptr, *shn = nullptr;
    Dd *eb = nullptr, *leg = nullptr;
    double* part = nullptr;
    unsigned* err = nullptr;
};
inline void want_eval(Scratch1& S, EvalBufs& B, int n) {
    const size_t N = (size_t)n, W = (size_t)ad_warps(n);
    S.want(&B.xf, sizeof(int4) * N);
    S.want(&B.shj, sizeof(int) * N * kAdCand);
    S.want(&B.shn, sizeof(int) * N);
    S.want(&B.eb, sizeof(Dd) * W * kAdComp * kAdEdges);
    S.want(&B.leg, sizeof(Dd) * N * kAdCand * 3);
    S.want(&B.part, sizeof(double) * W * kRed);
    S.want(&B.err, sizeof(unsigned));
}

FracArgs frac_args(const double box[3], double skin, int force) {
    FracArgs F;
    for (int k = 0; k < 3; ++k) {
        F.iL[k] = 1.0 / box[k];
        F.Lf[k] = (float)(box[k] * 0x1p-32);
    }
    // two atoms may each move half the skin before a pair outside the list can enter the cutoff;
    // the margin covers the rounding of the positions and of this test
    const double thr = 0.5 * skin - 1e-4;
    F.thr2 = thr > 0.0 ? (float)(thr * thr) : -1.0f;
    F.force = force;
    return F;
}

struct ListRef {
    int4* xf_ref = nullptr;      // fractional positions at the last build, and the rebuild flag
    int* rebuild = nullptr;
};

template <typename T, typename TP, bool GRAD>
void run_eval(const double* x, const double* w, int n, const double box[3], const int* nbr, const int* cnt, int cap,
              const SWp<TP>& P, double* f, double* fd, const EvalBufs& B, const ListRef& R, unsigned* err, cudaStream_t s) {
    AdArgs<T, TP> A;
    A.x = x; A.w = w; A.n = n; A.apw = atoms_per_warp(n);
    const FracArgs F = frac_args(box, 0.0, 0);
    for (int k = 0; k < 3; ++k) { A.L[k] = box[k]; A.iL[k] = F.iL[k]; A.Lf[k] = F.Lf[k]; }
    A.rcf2 = (float)P.rc2 * (1.0f + 1e-5f);
    A.xf = B.xf; A.xf_ref = R.xf_ref; A.rebuild = R.rebuild;
    A.nbr = nbr; A.cnt = cnt; A.cap = cap;
    A.row4 = (cap & 3) == 0 && (reinterpret_cast<uintptr_t>(nbr) & 15) == 0;
    A.P = P; A.shj = B.shj; A.shn = B.shn;
    A.eb = reinterpret_cast<T*>(B.eb); A.leg = reinterpret_cast<T*>(B.leg);
    A.part = B.part; A.err = err;
    k_sw_edges<T, TP, GRAD><<<ad_warps(n), 32, 0, s>>>(A);
    k_sw_gather<T><<<(4 * n + kAdThreads - 1) / kAdThreads, kAdThreads, 0, s>>>(n, B.shj, B.shn, A.leg, f, fd, err,
                                                                               R.rebuild);
}

// ---------------------------------------------------------------------------- integrator parts
// Per-step constants of the update, in FP64.
struct StepC {
    double c;      // dt / (2 m)
    double dt;
    double gm;     // m / tdamp (0 without thermostat)
    double amp;    // sqrt(2 m kB T / (tdamp dt)) (0 without thermostat)
    double kE;
    double s_int, s_E;   // force scales at the step's lambda
    double inv_n;
};

// vh = v + c F; x += dt vh (and the same for the tangents when X != NULL); the new positions'
// fractional form and list test, and a copy of the positions in keep (or NULL).
__global__ void __launch_bounds__(kAdThreads) k_half_drift(int n, StepC C, FracArgs Fa, double* x, const double* v,
                                                           const double* F, double* vh, double* X, const double* V,
                                                           const double* Fd, double* VH, double* keep, int4* xf,
                                                           const int4* ref, int* rebuild) {
    const int i = blockIdx.x * kAdThreads + threadIdx.x;
    if (i >= n) return;
    double xn[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const size_t t = (size_t)k * n + i;
        const double h = v[t] + C.c * F[t];
        vh[t] = h;
        xn[k] = x[t] + C.dt * h;
        x[t] = xn[k];
        if (keep) keep[t] = xn[k];
        if (X) {
            const double H = V[t] + C.c * Fd[t];
            VH[t] = H;
            X[t] = X[t] + C.dt * H;
        }
    }
    frac_atom(Fa, i, xn, xf, ref, rebuild);
}

// Per-block sums of the noise (3 components), of |x - r0|^2 and of (x - r0) . X.
__global__ void __launch_bounds__(kAdThreads) k_noise_spring_part(int n, const double* xi_aos, const double* x,
                                                                  const double* r0, const double* X, double* part) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    double v[kRed];
    for (int k = 0; k < kRed; ++k) v[k] = 0.0;
    if (i < n) {
        const size_t N = (size_t)n;
        for (int k = 0; k < 3; ++k) {
            if (xi_aos) v[k] = xi_aos[3 * i + k];
            if (r0) {
                const double d = x[k * N + i] - r0[k * N + i];
                v[3] += d * d;
                if (X) v[4] += d * X[k * N + i];
            }
        }
    }
    warp_block_sum(v, r0 ? (X ? 5 : 4) : 3, part + (size_t)blockIdx.x * kRed);
}

// Work scalars on the device.
struct Scal {
    double sw[kRed];     // last SW evaluation [E, E', G(7), G'(7)]
    double ns[kRed];     // last noise / spring sums
    double W, dW;
    double th[7];        // accumulated dW/dtheta (reverse sweep)
};

// Work increment of a step: W += D dl with D = U_E - U (FL) or U + P V (RS); dW += D' dl.
struct WorkC {
    int kind, add;
    double kE, PV, dl;
};

// F = s_int F_sw + s_E (-kE (x - r0)) - gm vh + amp (xi - mean xi); v = vh + c F (and the
// tangents); the first thread adds the work increment.
__global__ void k_finish(int n, StepC C, WorkC Wc, const double* fsw, const double* x, const double* r0, const double* vh,
                         const double* xi_aos, Scal* S, double* F, double* v,
                         const double* fswd, const double* X, const double* VH, double* Fd, double* V) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t == 0 && Wc.add) {
        const double ue = 0.5 * Wc.kE * S->ns[3], ued = Wc.kE * S->ns[4];
        const bool fl = Wc.kind == NEFE_SCHED_FL;
        const double D = fl ? ue - S->sw[0] : S->sw[0] + Wc.PV, Dt = fl ? ued - S->sw[1] : S->sw[1];
        S->W += D * Wc.dl;
        S->dW += Dt * Wc.dl;
    }
    if (t >= 3 * n) return;
    const int k = t / n, i = t - k * n;
    double f = C.s_int * fsw[t] - C.gm * vh[t];
    if (r0 && C.s_E != 0.0) f -= C.s_E * C.kE * (x[t] - r0[t]);
    if (xi_aos) f += C.amp * (xi_aos[3 * i + k] - S->ns[k] * C.inv_n);
    F[t] = f;
    v[t] = vh[t] + C.c * f;
    if (Fd) {
        double g = C.s_int * fswd[t] - C.gm * VH[t];
        if (r0 && C.s_E != 0.0) g -= C.s_E * C.kE * X[t];
        Fd[t] = g;
        V[t] = VH[t] + C.c * g;
    }
}

// Reverse sweep, before the evaluation at x = x_{k+1}: w = fb + c vb (adjoint of F_{k+1}), and x's
// fractional form and list test.
__global__ void __launch_bounds__(kAdThreads) k_rev_pre(int n, double c, FracArgs Fa, const double* fb, const double* vb,
                                                        double* w, const double* x, int4* xf, const int4* ref,
                                                        int* rebuild) {
    const int i = blockIdx.x * kAdThreads + threadIdx.x;
    if (i >= n) return;
    double xx[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const size_t t = (size_t)k * n + i;
        w[t] = fb[t] + c * vb[t];
        xx[k] = x[t];
    }
    frac_atom(Fa, i, xx, xf, ref, rebuild);
}

// Reverse sweep after the evaluation at x_{k+1} (fsw, fswd = J w there):
//   xb += s_int J w - s_E kE w + dl grad_x D(x_{k+1});  vh_b = vb - gm w + dt xb;  vb = vh_b;  fb = c vh_b;
//   th += s_int (dF/dtheta)^T w + dl dD/dtheta = -s_int G' + dl (-G for FL, +G for RS).
// With final != 0 (the evaluation at x_0) it writes dW/dx0 into xb and dW/dv0 into vb instead.
__global__ void k_rev_post(int n3, StepC C, int kind, double dl, const double* x, const double* r0,
                           const double* fsw, const double* fswd, const double* w, double* xb, double* vb,
                           double* fb, int final_, Scal* S) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t < 7) {
        const double G = S->sw[2 + t], Gd = S->sw[9 + t];
        S->th[t] += -C.s_int * Gd + dl * (kind == NEFE_SCHED_FL ? -G : G);
    }
    if (t >= n3) return;
    double gD;
    if (kind == NEFE_SCHED_FL) gD = (r0 ? C.kE * (x[t] - r0[t]) : 0.0) + fsw[t];
    else gD = -fsw[t];
    double xbn = xb[t] + C.s_int * fswd[t] + dl * gD;
    if (r0 && C.s_E != 0.0) xbn -= C.s_E * C.kE * w[t];
    if (final_) {
        xb[t] = xbn;
        vb[t] = vb[t] - C.gm * w[t];
        return;
    }
    const double vh = vb[t] - C.gm * w[t] + C.dt * xbn;
    xb[t] = xbn;
    vb[t] = vh;
    fb[t] = C.c * vh;
}

inline int eblocks(long n) { return (int)((n + 255) / 256); }

}  // namespace ad
}  // namespace nefe

using namespace nefe;
using namespace nefe::ad;

// ---------------------------------------------------------------------------- adjoint context
struct nefe_adj {
    int device = 0;
    cudaStream_t s = nullptr;
    nefe_adjoint_desc d;
    nefe_sw_params prm;
    int n = 0;
    double rcs = 0;
    double PV = 0;
    long nsteps = 0;          // length of the last forward run
    std::vector<double> lam;  // lambda_0 .. lambda_K
    Scratch1 L;               // list build, evaluation scratch
    Bufs lb;
    EvalBufs B;
    ListRef R;                // where the lists were built, and the flag that they are stale
    int *rtiles = nullptr, *rcount = nullptr, *rcbase = nullptr;
    bool force_list = true;   // the next evaluation builds the lists whatever the displacements
    // device arrays (SoA [3n] unless noted)
    double *x0 = nullptr, *v0 = nullptr, *r0 = nullptr;
    double *x = nullptr, *v = nullptr, *F = nullptr, *vh = nullptr, *fsw = nullptr, *fswd = nullptr;
    double *X = nullptr, *V = nullptr, *Fd = nullptr, *VH = nullptr;
    double *xb = nullptr, *vb = nullptr, *fb = nullptr, *w = nullptr;
    double* xi = nullptr;     // AoS [n][3] noise of one step
    double* part = nullptr;   // [nblocks][kRed] noise and spring sums
    double* ckpt = nullptr;   // [nckpt][3][3n]: x, v, F
    double* seg = nullptr;    // [K_c][3n] positions x_{k+1} of one segment
    long nckpt = 0;
    int* nbr = nullptr;
    int* cnt = nullptr;
    Scal* S = nullptr;
    unsigned* err = nullptr;
    std::vector<void*> owned;

    template <typename P>
    cudaError_t alloc(P** p, size_t bytes) {
        void* q = nullptr;
        cudaError_t e = device_alloc(&q, bytes < 16 ? 16 : bytes);
        if (e == cudaSuccess) owned.push_back(q);
        *p = static_cast<P*>(q);
        return e;
    }
    ~nefe_adj() {
        for (void* p : owned) cudaFree(p);
    }
};

namespace {

double sched_lambda_host(const nefe_adjoint_desc& d, long k) {
    double tau = d.nsched > 0 ? (double)k / (double)d.nsched : 1.0;
    if (tau > 1.0) tau = 1.0;
    if (d.direction < 0) tau = 1.0 - tau;
    if (d.kind == NEFE_SCHED_FL) {
        const double t2 = tau * tau, t4 = t2 * t2;
        return tau * t4 * (70.0 * t4 - 315.0 * t2 * tau + 540.0 * t2 - 420.0 * tau + 126.0);
    }
    return 1.0 / (1.0 + tau * (1.0 / d.lambda_f - 1.0));
}

StepC step_consts(const nefe_adj* A, long k) {
    StepC C;
    const double me = A->d.mass * kMvv2e;
    C.c = 0.5 * A->d.dt / me;
    C.dt = A->d.dt;
    const bool th = A->d.tdamp > 0.0;
    C.gm = th ? me / A->d.tdamp : 0.0;
    C.amp = th ? std::sqrt(2.0 * me * kB * A->d.T / (A->d.tdamp * A->d.dt)) : 0.0;
    C.kE = A->d.k_E;
    const double l = A->lam[(size_t)k];
    if (A->d.kind == NEFE_SCHED_FL) { C.s_int = 1.0 - l; C.s_E = l; }
    else { C.s_int = l; C.s_E = 0.0; }
    C.inv_n = 1.0 / (double)A->n;
    return C;
}

// Fractional form and list test of the next evaluation's positions.
FracArgs frac_of(nefe_adj* A) {
    const FracArgs F = frac_args(A->d.box, A->rcs - A->prm.a * A->prm.sigma, A->force_list ? 1 : 0);
    A->force_list = false;
    return F;
}

// SW evaluation at x, whose fractional form is in A->B.xf; the lists are rebuilt there if some atom
// is more than half the skin from where they were built (the kernels of the build return at once
// otherwise).  A pair outside the cutoff contributes nothing, so the result does not depend on
// when the lists were built.  mode 0: energy and forces; 1: tangents along w and dth; 2: products
// along w and the parameter derivatives.
void eval_at(nefe_adj* A, const double* x, const double* w, const double* dth, int mode) {
    A->lb.x = const_cast<double*>(x);
    launch_cells_and_list(A->lb, NEFE_FP32, (A->n + kTile - 1) / kTile, 1, 0, A->s, nullptr);
    const double* box = A->d.box;
    if (mode == 0)
        run_eval<double, double, false>(x, nullptr, A->n, box, A->nbr, A->cnt, A->d.nbr_cap, sw_params_real(A->prm), A->fsw,
                                        nullptr, A->B, A->R, A->err, A->s);
    else if (mode == 1)
        run_eval<Dd, Dd, false>(x, w, A->n, box, A->nbr, A->cnt, A->d.nbr_cap, sw_params_dual(A->prm, dth), A->fsw, A->fswd,
                                A->B, A->R, A->err, A->s);
    else
        run_eval<Dd, double, true>(x, w, A->n, box, A->nbr, A->cnt, A->d.nbr_cap, sw_params_real(A->prm), A->fsw, A->fswd,
                                   A->B, A->R, A->err, A->s);
}

// Noise of step `step` and spring sums at x; the evaluation's and these sums; then F, v (and
// tangents) and the work increment by k_finish.
void finish_at(nefe_adj* A, long step, const double* vsrc_half, bool tangent, bool work) {
    const int n = A->n;
    const bool th = A->d.tdamp > 0.0;
    if (th) launch_noise(A->d.seed, A->d.sys_id, (unsigned long long)step, n, NEFE_FP64, A->xi, A->s);
    const int nb = ad_blocks(n);
    k_noise_spring_part<<<nb, kAdThreads, 0, A->s>>>(n, th ? A->xi : nullptr, A->x, A->r0,
                                                       tangent ? A->X : nullptr, A->part);
    k_sum_rows<<<2 * kRed, 128, 0, A->s>>>(A->B.part, ad_warps(n), A->S->sw, A->part, nb, A->S->ns);
    const StepC C = step_consts(A, step);
    WorkC W{A->d.kind, work && step < A->nsteps ? 1 : 0, A->d.k_E, A->PV, 0.0};
    if (W.add) W.dl = A->lam[(size_t)step + 1] - A->lam[(size_t)step];
    k_finish<<<eblocks(3L * n), 256, 0, A->s>>>(n, C, W, A->fsw, A->x, A->r0, vsrc_half, th ? A->xi : nullptr,
                                                A->S, A->F, A->v, tangent ? A->fswd : nullptr,
                                                tangent ? A->X : nullptr, tangent ? A->VH : nullptr,
                                                tangent ? A->Fd : nullptr, tangent ? A->V : nullptr);
}

// Initial force at step 0 (damping on v0, noise with step counter 0), from x = x0, v = v0.
void setup_run(nefe_adj* A, bool tangent, const double* dth) {
    const size_t b3 = sizeof(double) * 3 * (size_t)A->n;
    cudaMemcpyAsync(A->x, A->x0, b3, cudaMemcpyDeviceToDevice, A->s);
    cudaMemcpyAsync(A->vh, A->v0, b3, cudaMemcpyDeviceToDevice, A->s);
    if (tangent) cudaMemcpyAsync(A->VH, A->V, b3, cudaMemcpyDeviceToDevice, A->s);
    A->force_list = true;
    k_frac<<<ad_blocks(A->n), kAdThreads, 0, A->s>>>(A->n, frac_of(A), A->x, A->B.xf, A->R.xf_ref, A->R.rebuild);
    eval_at(A, A->x, tangent ? A->X : nullptr, dth, tangent ? 1 : 0);
    finish_at(A, 0, A->vh, tangent, true);
    // finish_at wrote v = vh + c F; the state after setup keeps v = v0
    cudaMemcpyAsync(A->v, A->v0, b3, cudaMemcpyDeviceToDevice, A->s);
    if (tangent) cudaMemcpyAsync(A->V, A->VH, b3, cudaMemcpyDeviceToDevice, A->s);
}

void drift(nefe_adj* A, long k, bool tangent, double* keep) {
    k_half_drift<<<ad_blocks(A->n), kAdThreads, 0, A->s>>>(
        A->n, step_consts(A, k), frac_of(A), A->x, A->v, A->F, A->vh, tangent ? A->X : nullptr, tangent ? A->V : nullptr,
        tangent ? A->Fd : nullptr, tangent ? A->VH : nullptr, keep, A->B.xf, A->R.xf_ref, A->R.rebuild);
}

// One step k -> k+1 of the trajectory (and of the tangents).
void step_run(nefe_adj* A, long k, bool tangent, const double* dth) {
    drift(A, k, tangent, nullptr);
    eval_at(A, A->x, tangent ? A->X : nullptr, dth, tangent ? 1 : 0);
    finish_at(A, k + 1, A->vh, tangent, true);
}

// One step of the reverse sweep: the adjoint variables through the evaluation at x = x_k.
void rev_at(nefe_adj* A, long k, const double* x, double dl, bool last) {
    const StepC C = step_consts(A, k);
    k_rev_pre<<<ad_blocks(A->n), kAdThreads, 0, A->s>>>(A->n, last ? 0.0 : C.c, frac_of(A), A->fb, A->vb, A->w, x, A->B.xf,
                                                         A->R.xf_ref, A->R.rebuild);
    eval_at(A, x, A->w, nullptr, 2);
    k_sum_rows<<<kRed, 128, 0, A->s>>>(A->B.part, ad_warps(A->n), A->S->sw, nullptr, 0, nullptr);
    k_rev_post<<<eblocks(3L * A->n), 256, 0, A->s>>>(3 * A->n, C, A->d.kind, dl, x, A->r0, A->fsw, A->fswd, A->w, A->xb,
                                                     A->vb, A->fb, last ? 1 : 0, A->S);
}

int read_errors(nefe_adj* A, const char* where) {
    unsigned e1 = 0;
    DevState st;
    NEFE_CU(cudaMemcpyAsync(&e1, A->err, sizeof(unsigned), cudaMemcpyDeviceToHost, A->s));
    NEFE_CU(cudaMemcpyAsync(&st, A->L.st, sizeof(st), cudaMemcpyDeviceToHost, A->s));
    NEFE_CU(cudaStreamSynchronize(A->s));
    NEFE_CU(cudaGetLastError());
    const unsigned e = e1 | st.err;
    if (e & NEFE_ERR_NBR_OVERFLOW) return fail(NEFE_EOVERFLOW, "%s: neighbour row above cap", where);
    if (e & NEFE_ERR_SHELL_OVERFLOW) return fail(NEFE_EOVERFLOW, "%s: shell above 32 neighbours", where);
    if (e & NEFE_ERR_NAN) return fail(NEFE_ENAN, "%s: non-finite energy or force", where);
    if (e) return fail(NEFE_EINVAL, "%s: error word 0x%x", where, e);
    return NEFE_OK;
}

int reset_errors(nefe_adj* A) {
    NEFE_CU(cudaMemsetAsync(A->err, 0, sizeof(unsigned), A->s));
    NEFE_CU(cudaMemsetAsync(reinterpret_cast<char*>(A->L.st) + offsetof(DevState, err), 0, sizeof(unsigned), A->s));
    return NEFE_OK;
}

int prepare_schedule(nefe_adj* A, long nsteps) {
    int rc = reset_errors(A);
    if (rc) return rc;
    A->nsteps = nsteps;
    A->lam.resize((size_t)nsteps + 1);
    for (long k = 0; k <= nsteps; ++k) A->lam[(size_t)k] = sched_lambda_host(A->d, k);
    const long kc = A->d.checkpoint_every;
    const long need = nsteps / kc + 1;
    if (need > A->nckpt) {
        if (A->ckpt) {
            NEFE_CU(cudaStreamSynchronize(A->s));
            for (auto it = A->owned.begin(); it != A->owned.end(); ++it)
                if (*it == A->ckpt) { A->owned.erase(it); break; }
            cudaFree(A->ckpt);
            A->ckpt = nullptr;
        }
        NEFE_CU(A->alloc(&A->ckpt, sizeof(double) * 9 * (size_t)A->n * (size_t)need));
        A->nckpt = need;
    }
    return NEFE_OK;
}

void save_ckpt(nefe_adj* A, long idx) {
    const size_t b3 = sizeof(double) * 3 * (size_t)A->n;
    double* c = A->ckpt + (size_t)idx * 9 * (size_t)A->n;
    cudaMemcpyAsync(c, A->x, b3, cudaMemcpyDeviceToDevice, A->s);
    cudaMemcpyAsync(c + 3 * (size_t)A->n, A->v, b3, cudaMemcpyDeviceToDevice, A->s);
    cudaMemcpyAsync(c + 6 * (size_t)A->n, A->F, b3, cudaMemcpyDeviceToDevice, A->s);
}

void load_ckpt(nefe_adj* A, long idx) {
    const size_t b3 = sizeof(double) * 3 * (size_t)A->n;
    const double* c = A->ckpt + (size_t)idx * 9 * (size_t)A->n;
    cudaMemcpyAsync(A->x, c, b3, cudaMemcpyDeviceToDevice, A->s);
    cudaMemcpyAsync(A->v, c + 3 * (size_t)A->n, b3, cudaMemcpyDeviceToDevice, A->s);
    cudaMemcpyAsync(A->F, c + 6 * (size_t)A->n, b3, cudaMemcpyDeviceToDevice, A->s);
}

int upload_aos(nefe_adj* A, const double* host, double* dev) {
    const size_t b3 = sizeof(double) * 3 * (size_t)A->n;
    NEFE_CU(cudaMemcpyAsync(A->w, host, b3, cudaMemcpyHostToDevice, A->s));
    launch_aos_soa(A->w, dev, A->n, 1, A->s);
    return NEFE_OK;
}

int download_aos(nefe_adj* A, const double* dev, double* host) {
    const size_t b3 = sizeof(double) * 3 * (size_t)A->n;
    launch_aos_soa(dev, A->w, A->n, 0, A->s);
    NEFE_CU(cudaMemcpyAsync(host, A->w, b3, cudaMemcpyDeviceToHost, A->s));
    return NEFE_OK;
}

}  // namespace

extern "C" {

int nefe_sw_dual(const double* x, const double* w, int n, const double box[3], double rcs, const int* nbr,
                 const int* cnt, int cap, const nefe_sw_params* prm, const double* dtheta, double* f,
                 double* fd, double* out16, void* stream) {
    NvtxRange nvtx_("nefe_sw_dual");
    if (n < 0 || !box || cap < 1 || cap > kMaxCap || !valid_params(prm) || !out16 ||
        (n > 0 && (!x || !nbr || !cnt || !f || !fd)))
        return fail(NEFE_EINVAL, "nefe_sw_dual: bad argument");
    if (prm->a * prm->sigma > rcs) return fail(NEFE_EINVAL, "nefe_sw_dual: a*sigma above rcs");
    int rc = check_box(box, rcs);
    if (rc) return rc;
    cudaStream_t s = (cudaStream_t)stream;
    if (n == 0) {
        NEFE_CU(cudaMemsetAsync(out16, 0, sizeof(double) * kRed, s));
        NEFE_CU(cudaStreamSynchronize(s));
        return NEFE_OK;
    }
    Scratch1 S;
    EvalBufs B;
    S.s = s;
    want_eval(S, B, n);
    NEFE_CU(S.commit());
    NEFE_CU(cudaMemsetAsync(B.err, 0, sizeof(unsigned), s));
    k_frac<<<ad_blocks(n), kAdThreads, 0, s>>>(n, frac_args(box, 0.0, 0), x, B.xf, nullptr, nullptr);
    if (dtheta)
        run_eval<Dd, Dd, true>(x, w, n, box, nbr, cnt, cap, sw_params_dual(*prm, dtheta), f, fd, B, ListRef{}, B.err, s);
    else
        run_eval<Dd, double, true>(x, w, n, box, nbr, cnt, cap, sw_params_real(*prm), f, fd, B, ListRef{}, B.err, s);
    k_sum_rows<<<kRed, 128, 0, s>>>(B.part, ad_warps(n), out16, nullptr, 0, nullptr);
    unsigned e = 0;
    NEFE_CU(cudaMemcpyAsync(&e, B.err, sizeof(unsigned), cudaMemcpyDeviceToHost, s));
    NEFE_CU(cudaStreamSynchronize(s));
    NEFE_CU(cudaGetLastError());
    if (e & NEFE_ERR_SHELL_OVERFLOW) return fail(NEFE_EOVERFLOW, "nefe_sw_dual: shell above 32 neighbours");
    if (e & NEFE_ERR_NAN) return fail(NEFE_ENAN, "nefe_sw_dual: non-finite energy or force");
    return NEFE_OK;
}

int nefe_adjoint_create(nefe_adj** out, int device, void* stream, const nefe_adjoint_desc* d,
                        const nefe_sw_params* prm) {
    if (!out || !d || !valid_params(prm) || d->n <= 0 || !d->x || !d->v || d->mass <= 0 || d->dt <= 0 ||
        d->nbr_cap < 1 || d->nbr_cap > kMaxCap || d->checkpoint_every < 1 || d->skin < 0 ||
        (d->kind != NEFE_SCHED_FL && d->kind != NEFE_SCHED_RS) || (d->direction != 1 && d->direction != -1) ||
        d->nsched < 1 || (d->kind == NEFE_SCHED_FL && (!d->r0 || d->k_E <= 0)) ||
        (d->kind == NEFE_SCHED_RS && !(d->lambda_f > 0)) || (d->tdamp > 0 && !(d->T > 0)))
        return fail(NEFE_EINVAL, "nefe_adjoint_create: bad argument");
    if (d->n >= (1 << kCodeShift)) return fail(NEFE_EINVAL, "nefe_adjoint_create: n above 2^27");
    *out = nullptr;
    NEFE_CU(cudaSetDevice(device));
    const double rcs = prm->a * prm->sigma + d->skin;
    int rc = check_box(d->box, rcs);
    if (rc) return rc;
    int n3[3];
    if (!host_grid(d->box, rcs, n3)) return fail(NEFE_EINVAL, "nefe_adjoint_create: fewer than 2 cells on an axis");
    nefe_adj* A = new nefe_adj();
    A->device = device;
    A->s = (cudaStream_t)stream;
    A->d = *d;
    A->prm = *prm;
    A->n = d->n;
    A->rcs = rcs;
    A->PV = d->P_GPa / kEvA3ToGPa * d->box[0] * d->box[1] * d->box[2];
    A->L.s = A->s;
    const int n = A->n;
    const size_t b3 = sizeof(double) * 3 * (size_t)n;
    auto bail = [&](int code) { cudaStreamSynchronize(A->s); delete A; return code; };
    want1(A->L, n, n3, NEFE_FP32, true);
    want_eval(A->L, A->B, n);
    A->L.want(&A->R.xf_ref, sizeof(int4) * (size_t)n);
    A->L.want(&A->rtiles, sizeof(int) * (size_t)((n + kTile - 1) / kTile));
    A->L.want(&A->rcount, sizeof(int));
    A->L.want(&A->rcbase, sizeof(int) * 2);
    if ((rc = commit1(A->L, n, d->box, rcs, n3, NEFE_FP32))) return bail(rc);
    A->R.rebuild = &A->L.st->rebuild;
    A->lb = bufs_of(A->L, nullptr, n);
    double** arrs[] = {&A->x0, &A->v0, &A->x, &A->v, &A->F, &A->vh, &A->fsw, &A->fswd, &A->X, &A->V, &A->Fd,
                       &A->VH, &A->xb, &A->vb, &A->fb, &A->w, &A->xi};
    for (double** p : arrs)
        if (A->alloc(p, b3) != cudaSuccess) return bail(fail(NEFE_ENOMEM, "nefe_adjoint_create: device memory"));
    if (d->r0 && A->alloc(&A->r0, b3) != cudaSuccess) return bail(fail(NEFE_ENOMEM, "nefe_adjoint_create: r0"));
    if (A->alloc(&A->part, sizeof(double) * kRed * (size_t)ad_blocks(n)) != cudaSuccess ||
        A->alloc(&A->seg, b3 * (size_t)d->checkpoint_every) != cudaSuccess ||
        A->alloc(&A->nbr, sizeof(int) * (size_t)n * d->nbr_cap) != cudaSuccess ||
        A->alloc(&A->cnt, sizeof(int) * (size_t)n) != cudaSuccess ||
        A->alloc(&A->S, sizeof(Scal)) != cudaSuccess || A->alloc(&A->err, sizeof(unsigned)) != cudaSuccess)
        return bail(fail(NEFE_ENOMEM, "nefe_adjoint_create: device memory"));
    A->lb.nbr = A->nbr; A->lb.cnt = A->cnt; A->lb.cap = d->nbr_cap;
    A->lb.rtiles = A->rtiles; A->lb.rcount = A->rcount; A->lb.rcbase = A->rcbase;
    if ((rc = upload_aos(A, d->x, A->x0)) || (rc = upload_aos(A, d->v, A->v0))) return bail(rc);
    if (d->r0 && (rc = upload_aos(A, d->r0, A->r0))) return bail(rc);
    if (cudaMemsetAsync(A->err, 0, sizeof(unsigned), A->s) != cudaSuccess ||
        cudaMemsetAsync(A->S, 0, sizeof(Scal), A->s) != cudaSuccess ||
        cudaStreamSynchronize(A->s) != cudaSuccess)
        return bail(cuda_fail(cudaGetLastError(), "nefe_adjoint_create"));
    A->d.x = A->d.v = A->d.r0 = nullptr;   // host arrays are not kept
    *out = A;
    return NEFE_OK;
}

int nefe_adjoint_set_params(nefe_adj* A, const nefe_sw_params* prm) {
    if (!A || !valid_params(prm)) return fail(NEFE_EINVAL, "nefe_adjoint_set_params: bad argument");
    if (prm->a * prm->sigma > A->rcs)
        return fail(NEFE_EINVAL, "nefe_adjoint_set_params: a*sigma above the list radius %g", A->rcs);
    A->prm = *prm;
    A->nsteps = 0;   // checkpoints belong to the old parameters
    return NEFE_OK;
}

int nefe_adjoint_destroy(nefe_adj* A) {
    if (!A) return NEFE_OK;
    cudaSetDevice(A->device);
    cudaStreamSynchronize(A->s);
    delete A;
    return NEFE_OK;
}

int nefe_adjoint_forward(nefe_adj* A, long nsteps, double* W) {
    NvtxRange nvtx_("nefe_adjoint_forward");
    if (!A || nsteps < 1) return fail(NEFE_EINVAL, "nefe_adjoint_forward: bad argument");
    NEFE_CU(cudaSetDevice(A->device));
    int rc = prepare_schedule(A, nsteps);
    if (rc) return rc;
    NEFE_CU(cudaMemsetAsync(A->S, 0, sizeof(Scal), A->s));
    setup_run(A, false, nullptr);
    save_ckpt(A, 0);
    const long kc = A->d.checkpoint_every;
    for (long k = 0; k < nsteps; ++k) {
        step_run(A, k, false, nullptr);
        if ((k + 1) % kc == 0 && k + 1 < nsteps) save_ckpt(A, (k + 1) / kc);
    }
    Scal h;
    NEFE_CU(cudaMemcpyAsync(&h, A->S, sizeof(h), cudaMemcpyDeviceToHost, A->s));
    rc = read_errors(A, "nefe_adjoint_forward");
    if (rc) return rc;
    if (W) *W = h.W;
    return NEFE_OK;
}

int nefe_adjoint_backward(nefe_adj* A, double dW_dtheta[7], double* dW_dx0, double* dW_dv0) {
    NvtxRange nvtx_("nefe_adjoint_backward");
    if (!A || !dW_dtheta) return fail(NEFE_EINVAL, "nefe_adjoint_backward: bad argument");
    if (A->nsteps < 1) return fail(NEFE_ESTATE, "nefe_adjoint_backward: run nefe_adjoint_forward first");
    NEFE_CU(cudaSetDevice(A->device));
    const size_t n3 = 3 * (size_t)A->n;
    const size_t b3 = sizeof(double) * n3;
    const long K = A->nsteps, kc = A->d.checkpoint_every;
    int rc0 = reset_errors(A);
    if (rc0) return rc0;
    NEFE_CU(cudaMemsetAsync(A->xb, 0, b3, A->s));
    NEFE_CU(cudaMemsetAsync(A->vb, 0, b3, A->s));
    NEFE_CU(cudaMemsetAsync(A->fb, 0, b3, A->s));
    NEFE_CU(cudaMemsetAsync(A->S->th, 0, sizeof(double) * 7, A->s));
    const long nseg = (K + kc - 1) / kc;
    A->force_list = true;
    for (long sg = nseg - 1; sg >= 0; --sg) {
        const long k0 = sg * kc, k1 = (k0 + kc < K) ? k0 + kc : K;
        // recompute the segment from its checkpoint, keeping x_{k+1}
        load_ckpt(A, sg);
        for (long k = k0; k < k1; ++k) {
            drift(A, k, false, A->seg + (size_t)(k - k0) * n3);
            if (k + 1 < k1) {
                eval_at(A, A->x, nullptr, nullptr, 0);
                finish_at(A, k + 1, A->vh, false, false);
            }
        }
        // step the adjoint variables back through the segment
        for (long k = k1 - 1; k >= k0; --k) {
            const double dl = (k + 1 < K) ? A->lam[(size_t)k + 2] - A->lam[(size_t)k + 1] : 0.0;
            rev_at(A, k + 1, A->seg + (size_t)(k - k0) * n3, dl, false);
        }
    }
    // the initial force F_0 = F(x_0) - gm v_0 + noise, and the work term at x_0
    rev_at(A, 0, A->x0, A->lam[1] - A->lam[0], true);
    Scal h;
    NEFE_CU(cudaMemcpyAsync(&h, A->S, sizeof(h), cudaMemcpyDeviceToHost, A->s));
    int rc = 0;
    if (dW_dx0 && (rc = download_aos(A, A->xb, dW_dx0))) return rc;
    if (dW_dv0 && (rc = download_aos(A, A->vb, dW_dv0))) return rc;
    rc = read_errors(A, "nefe_adjoint_backward");
    if (rc) return rc;
    for (int k = 0; k < 7; ++k) dW_dtheta[k] = h.th[k];
    return NEFE_OK;
}

int nefe_adjoint_tangent(nefe_adj* A, long nsteps, const double dtheta[7], const double* dx0,
                         const double* dv0, double* W, double* dW) {
    NvtxRange nvtx_("nefe_adjoint_tangent");
    if (!A || nsteps < 1 || !dtheta) return fail(NEFE_EINVAL, "nefe_adjoint_tangent: bad argument");
    NEFE_CU(cudaSetDevice(A->device));
    const size_t b3 = sizeof(double) * 3 * (size_t)A->n;
    int rc = prepare_schedule(A, nsteps);
    if (rc) return rc;
    NEFE_CU(cudaMemsetAsync(A->S, 0, sizeof(Scal), A->s));
    if (dx0) { if ((rc = upload_aos(A, dx0, A->X))) return rc; }
    else NEFE_CU(cudaMemsetAsync(A->X, 0, b3, A->s));
    if (dv0) { if ((rc = upload_aos(A, dv0, A->V))) return rc; }
    else NEFE_CU(cudaMemsetAsync(A->V, 0, b3, A->s));
    setup_run(A, true, dtheta);
    for (long k = 0; k < nsteps; ++k) step_run(A, k, true, dtheta);
    Scal h;
    NEFE_CU(cudaMemcpyAsync(&h, A->S, sizeof(h), cudaMemcpyDeviceToHost, A->s));
    rc = read_errors(A, "nefe_adjoint_tangent");
    A->nsteps = 0;   // no checkpoints of this run: a backward needs a forward first
    if (rc) return rc;
    if (W) *W = h.W;
    if (dW) *dW = h.dW;
    return NEFE_OK;
}

int nefe_adjoint_state(nefe_adj* A, double* x, double* v) {
    if (!A) return fail(NEFE_EINVAL, "nefe_adjoint_state: bad argument");
    NEFE_CU(cudaSetDevice(A->device));
    int rc = 0;
    if (x && (rc = download_aos(A, A->x, x))) return rc;
    if (v && (rc = download_aos(A, A->v, v))) return rc;
    NEFE_CU(cudaStreamSynchronize(A->s));
    return NEFE_OK;
}

}  // extern "C"
