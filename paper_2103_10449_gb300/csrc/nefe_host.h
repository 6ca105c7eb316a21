// Host helpers shared by the C-ABI translation units of libnefe.
#pragma once
#include <cuda_runtime.h>
#include <cmath>
#include <utility>
#include <vector>

#include "nefe.h"
#include "nefe_dev.h"
#include "nefe_launch.h"

namespace nefe {

// Records a message for nefe_last_error() and returns code.
int fail(int code, const char* fmt, ...);
// Maps a CUDA error to NEFE_ECUDA with a message (NEFE_OK when e == cudaSuccess).
int cuda_fail(cudaError_t e, const char* where);

#define NEFE_CU(call)                                   \
    do {                                                \
        cudaError_t e_ = (call);                        \
        if (e_ != cudaSuccess) return cuda_fail(e_, #call); \
    } while (0)

// Cell grid of the list-build rule (same arithmetic as the device): floor(L/rcs), reduced
// while L/n < rcs (1 + 1e-9).  Returns false when an axis gets fewer than 2 cells.
inline bool host_grid(const double box[3], double rcs, int n3[3]) {
    bool ok = true;
    for (int k = 0; k < 3; ++k) {
        // clamped before the conversion to int (a huge box would overflow it); so many cells
        // exceed every capacity and are rejected by the callers' cell-count check
        const double q = std::floor(box[k] / rcs);
        int m = q < (double)(1 << 20) ? (int)q : (1 << 20);
        while (m > 0 && box[k] / (double)m < rcs * (1.0 + 1e-9)) --m;
        if (m < 2) ok = false;
        n3[k] = m < 2 ? 2 : m;
    }
    return ok;
}

// The device side's reduction of a grid above the cell capacity: the longest axis loses cells
// (wider cells stay valid).
inline void cap_grid(int n3[3], long long cap) {
    while ((long long)n3[0] * n3[1] * n3[2] > cap) {
        const int k = (n3[0] >= n3[1] && n3[0] >= n3[2]) ? 0 : (n3[1] >= n3[2] ? 1 : 2);
        if (n3[k] <= 2) break;
        --n3[k];
    }
}

// Box and cell grid of a one-system state (the stateless calls; the engine sets them on the
// device when a list is built).
inline void set_grid(DevState& st, const double box[3], const int n3[3]) {
    for (int k = 0; k < 3; ++k) {
        st.box[k] = box[k];
        st.ncell[k] = n3[k];
        st.h[k] = st.hb[k] = box[k] / (double)n3[k];
        st.ibox[k] = 1.0 / box[k];
        st.h_f[k] = st.hb_f[k] = (float)st.h[k];
        st.rho_f[k] = 1.0f;
    }
    st.hmoved = 0;
    st.nbuild = 1;
}

inline int frac_fine(const double box[3]) { return std::fmax(box[0], std::fmax(box[1], box[2])) > kFracCoarse ? 1 : 0; }

// Power of two by which the scatter form's force unit is finer than silicon's (eps/sigma = 1.035, in
// the middle of an octave, so that fitted parameters keep the unit).
inline int leg_power(const nefe_sw_params& p) {
    const double force = p.eps / p.sigma * (1.4142135623730951 / 1.035);
    const int k = force > 0.0 && std::isfinite(force) ? -std::ilogb(force) : 0;
    return k < -60 ? -60 : (k > 60 ? 60 : k);
}

template <typename T>
inline SWc<T> make_swc(const nefe_sw_params& p) {
    SWc<T> c{};
    c.inv_sig = (T)(1.0 / p.sigma);
    c.a = (T)p.a;
    const double rc = p.a * p.sigma;
    c.rc2 = (T)(rc * rc);
    c.epsA = (T)(p.eps * p.A);
    c.B = (T)p.B;
    c.p = (T)p.p;
    c.q = (T)p.q;
    c.epslam = (T)(p.eps * p.lambda3);
    c.gam = (T)p.gamma;
    c.c0 = (T)p.cos0;
    c.eps = (T)p.eps;
    c.A = (T)p.A;
    c.lam3 = (T)p.lambda3;
    c.inv_sig_lo = (T)(1.0 / p.sigma - (double)c.inv_sig);
    c.a_lo = (T)(p.a - (double)c.a);
    c.B_lo = (T)(p.B - (double)c.B);
    // FP32 path: an edge whose three-body factor exp(gamma/(s - a)) is below 1e-12 adds forces
    // of order 1e-8 eV/A (pair and triplet), far below FP32 resolution, so it is dropped:
    // s_act = a + gamma / ln(1e-12).  FP64 path: only the last 1e-12 sigma before the cutoff
    // (where the terms underflow to 0) is dropped.
    if (sizeof(T) == 4) c.s_act = (T)(p.a + p.gamma / std::log(1e-12));
    else c.s_act = (T)(p.a - 1e-12);
    const double ract = (double)c.s_act * p.sigma;
    c.act2 = (T)(ract * ract < rc * rc ? ract * ract : rc * rc);
    c.int_pq = (p.p == 4.0 && p.q == 0.0) ? 1 : 0;
    c.leg_scale = (T)std::ldexp(kLegScale, leg_power(p));
    c.leg_fine = (T)std::ldexp(kLegFine, -leg_power(p));
    return c;
}

bool valid_params(const nefe_sw_params* p);

// Uhlenbeck-Ford constants of a system (mode UF_INT or UF_REF; list radius rc + skin).
inline void fill_uf(DevSys& d, const nefe_uf_params& uf, double skin, int mode) {
    const double kT = kB * uf.T;
    const double R = uf.rc + skin;
    d.uf_mode = mode;
    d.uf_pk = uf.p * kT;
    d.uf_is2 = 1.0 / (uf.sigma * uf.sigma);
    d.uf_rc2 = uf.rc * uf.rc;
    d.uf_shift = -d.uf_pk * std::log(-std::expm1(-d.uf_rc2 * d.uf_is2));
    d.uf_R2 = R * R;
    d.uf_pk_f = (float)d.uf_pk;
    d.uf_is2_f = (float)d.uf_is2;
    d.uf_rc2_f = (float)d.uf_rc2;
    d.uf_shift_f = (float)d.uf_shift;
    d.uf_R2_f = (float)d.uf_R2;
}
inline bool valid_uf(const nefe_uf_params* u) {
    return u && u->p > 0.0 && u->sigma > 0.0 && u->T > 0.0 && u->rc > 0.0 && std::isfinite(u->p) &&
           std::isfinite(u->sigma) && std::isfinite(u->T) && std::isfinite(u->rc);
}

// Stream-ordered device scratch from the library's own memory pool of the current device.
cudaError_t scratch_alloc(void** p, size_t bytes, cudaStream_t s);
// Gives the pools of all devices back (what is still allocated from them, once it is freed).
cudaError_t scratch_release();
// cudaMalloc, which takes back what the pools keep where the device is full.
cudaError_t device_alloc(void** p, size_t bytes);

// Single-system descriptors and scratch for the stateless calls and the adjoint context: the
// arrays are collected with want() and carved out of one stream-ordered allocation by commit(),
// which is released on the same stream.
struct Scratch1 {
    DevSys* sys = nullptr;
    DevState* st = nullptr;
    int4* tiles = nullptr;
    long long* acc = nullptr;
    void* swc = nullptr;
    int4* q = nullptr;
    void* xs = nullptr;
    void* xa = nullptr;
    void* xcs = nullptr;
    void* shd = nullptr;
    int* shj = nullptr;
    int* shn = nullptr;
    void* P = nullptr;
    int* cell_of = nullptr;
    int* perm = nullptr;
    int* cell_start = nullptr;
    int* cell_count = nullptr;
    int* cell_cursor = nullptr;
    int* scan_sums = nullptr;
    int4* xf = nullptr;
    int *lacc = nullptr, *hi_flag = nullptr;
    long long* lacc_hi = nullptr;
    float4* lscale = nullptr;
    uint2* xc = nullptr;
    int ncells = 0;
    cudaStream_t s = nullptr;
    void* base = nullptr;
    std::vector<std::pair<void**, size_t>> wanted;   // pointer to set, offset
    size_t total = 0;

    template <typename P>
    void want(P** p, size_t bytes) {
        wanted.emplace_back(reinterpret_cast<void**>(p), total);
        total += (bytes + 255) / 256 * 256;
    }
    cudaError_t commit() {
        const cudaError_t e = scratch_alloc(&base, total, s);
        for (auto& w : wanted) *w.first = e == cudaSuccess ? static_cast<char*>(base) + w.second : nullptr;
        return e;
    }
    ~Scratch1() {
        if (base) cudaFreeAsync(base, s);
    }
};

// NEFE_OK when every box length is positive, finite and at least 2 rcs.
int check_box(const double box[3], double rcs);
// Collects the one-system descriptors, the tile table, the sums and (cells) the cell arrays in S.
void want1(Scratch1& S, int n, const int n3[3], int prec, bool cells);
// Allocates what was collected and writes the descriptors, the tile table and zeroed sums and cell
// counts with one kernel (arguments by value: no copy from host memory).  With prm, the potential
// constants of precision prec go to S.swc; with uf, the system carries a Uhlenbeck-Ford term as
// U_int (list radius uf->rc + skin).
int commit1(Scratch1& S, int n, const double box[3], double rcs, const int n3[3], int prec,
            const nefe_sw_params* prm = nullptr, const nefe_uf_params* uf = nullptr, double skin = 0.0);
// Launch arguments over S for n atoms at FP64 positions x.
Bufs bufs_of(const Scratch1& S, const double* x, int n);

}  // namespace nefe
