// Stateless C-ABI entry points of libnefe (caller-owned device buffers) and error reporting.
#include <algorithm>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <mutex>
#include <shared_mutex>
#include <vector>

#include "nefe.h"
#include "nefe_dev.h"
#include "nefe_host.h"
#include "nefe_launch.h"
#include "nefe_nvtx.h"

namespace nefe {

static thread_local char g_msg[512] = "no error";

int fail(int code, const char* fmt, ...) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(g_msg, sizeof(g_msg), fmt, ap);
    va_end(ap);
    return code;
}

int cuda_fail(cudaError_t e, const char* where) {
    if (e == cudaSuccess) return NEFE_OK;
    if (e == cudaErrorMemoryAllocation) {
        cudaGetLastError();
        return fail(NEFE_ENOMEM, "%s: %s", where, cudaGetErrorString(e));
    }
    return fail(NEFE_ECUDA, "%s: %s", where, cudaGetErrorString(e));
}

bool valid_params(const nefe_sw_params* p) {
    return p && p->sigma > 0.0 && p->a > 0.0 && p->eps > 0.0 && std::isfinite(p->A) &&
           std::isfinite(p->B) && std::isfinite(p->p) && std::isfinite(p->q) &&
           std::isfinite(p->lambda3) && std::isfinite(p->gamma) && std::isfinite(p->cos0);
}

int check_box(const double box[3], double rcs) {
    for (int k = 0; k < 3; ++k)
        if (!(box[k] > 0.0) || !std::isfinite(box[k]))
            return fail(NEFE_EINVAL, "box length %d is not positive and finite", k);
    if (!(rcs > 0.0)) return fail(NEFE_EINVAL, "rcs must be positive");
    for (int k = 0; k < 3; ++k)
        if (box[k] < 2.0 * rcs)
            return fail(NEFE_EINVAL, "box length %g below 2*rcs = %g", box[k], 2.0 * rcs);
    return NEFE_OK;
}

// The library's scratch pool of a device.  The default pool hands its memory back to the driver
// at every synchronisation, so each call mapped its scratch anew (457 -> 207 us for a waited-for
// list and force call of 1723 atoms); this one keeps up to kScratchKeep bytes mapped between calls
// (anything above goes back at the next synchronisation) until nefe_release_scratch, or until an
// allocation of the library finds the device full.  Allocation and release are stream ordered, so
// calls on several streams and threads share it safely; the lock keeps a pool from being destroyed
// between its look-up and its use (what is allocated from it then stays valid until it is freed).
constexpr uint64_t kScratchKeep = 256ull << 20;
constexpr int kPoolDevices = 64;

static std::shared_mutex g_pool_mu;
static cudaMemPool_t g_pool[kPoolDevices] = {};

static cudaError_t make_pool(int dev) {
    std::unique_lock<std::shared_mutex> lock(g_pool_mu);
    if (g_pool[dev]) return cudaSuccess;
    cudaMemPoolProps props;
    std::memset(&props, 0, sizeof(props));
    props.allocType = cudaMemAllocationTypePinned;
    props.handleTypes = cudaMemHandleTypeNone;
    props.location.type = cudaMemLocationTypeDevice;
    props.location.id = dev;
    cudaMemPool_t pool = nullptr;
    cudaError_t e = cudaMemPoolCreate(&pool, &props);
    if (e != cudaSuccess) return e;
    uint64_t keep = kScratchKeep;
    e = cudaMemPoolSetAttribute(pool, cudaMemPoolAttrReleaseThreshold, &keep);
    if (e == cudaSuccess) g_pool[dev] = pool;
    else cudaMemPoolDestroy(pool);
    return e;
}

cudaError_t scratch_release() {
    std::unique_lock<std::shared_mutex> lock(g_pool_mu);
    cudaError_t first = cudaSuccess;
    for (cudaMemPool_t& pool : g_pool) {
        if (!pool) continue;
        const cudaError_t e = cudaMemPoolDestroy(pool);
        if (e != cudaSuccess && first == cudaSuccess) first = e;
        pool = nullptr;
    }
    return first;
}

cudaError_t scratch_alloc(void** p, size_t bytes, cudaStream_t s) {
    *p = nullptr;
    if (bytes < 16) bytes = 16;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return e;
    if (dev >= kPoolDevices) return cudaMallocAsync(p, bytes, s);
    for (;;) {
        {
            std::shared_lock<std::shared_mutex> lock(g_pool_mu);
            if (g_pool[dev]) return cudaMallocFromPoolAsync(p, bytes, g_pool[dev], s);
        }
        if ((e = make_pool(dev)) != cudaSuccess) return e;
    }
}

cudaError_t device_alloc(void** p, size_t bytes) {
    cudaError_t e = cudaMalloc(p, bytes);
    if (e != cudaErrorMemoryAllocation) return e;
    cudaGetLastError();
    scratch_release();                           // what the pool kept may be what is missing
    return cudaMalloc(p, bytes);
}

namespace {
struct SwcBytes {
    alignas(16) unsigned char b[sizeof(SWc<float>)];
};

__device__ __forceinline__ void copy_words(void* dst, const void* src, int bytes, int t) {
    if (4 * t < bytes) static_cast<unsigned*>(dst)[t] = static_cast<const unsigned*>(src)[t];
}

__global__ void __launch_bounds__(256) k_scratch_init(const __grid_constant__ DevSys hs, const __grid_constant__ DevState st,
                                                      const __grid_constant__ SwcBytes swc, DevSys* dsys, DevState* dst,
                                                      void* dswc, int4* tiles, int ntiles, long long* acc, int nacc,
                                                      int* counts, int ncells) {
    const int t = blockIdx.x * blockDim.x + threadIdx.x, stride = gridDim.x * blockDim.x;
    static_assert(sizeof(DevSys) <= 1024 && sizeof(DevState) <= 1024, "one word per thread of the first block");
    copy_words(dsys, &hs, (int)sizeof(hs), t);
    copy_words(dst, &st, (int)sizeof(st), t);
    copy_words(dswc, &swc, (int)sizeof(swc), t);
    for (int i = t; i < ntiles; i += stride) tiles[i] = make_int4(0, i * kTile, min(kTile, hs.n - i * kTile), 0);
    for (int i = t; i < nacc; i += stride) acc[i] = 0;
    for (int i = t; i < ncells; i += stride) counts[i] = 0;
}
}  // namespace

void want1(Scratch1& S, int n, const int n3[3], int prec, bool cells) {
    const size_t ntiles = (size_t)(n + kTile - 1) / kTile, N = (size_t)n;
    S.ncells = cells ? n3[0] * n3[1] * n3[2] : 0;
    S.want(&S.sys, sizeof(DevSys));
    S.want(&S.st, sizeof(DevState));
    S.want(&S.tiles, sizeof(int4) * (ntiles > 0 ? ntiles : 1));
    S.want(&S.acc, sizeof(long long) * 2 * ACC_N * kSlots);     // sums, then their remainders
    S.want(&S.swc, sizeof(SwcBytes));
    const size_t v4 = prec == NEFE_FP64 ? sizeof(double4) : sizeof(float4);
    if (cells || prec == NEFE_FP64) S.want(&S.xs, v4 * N);      // (the FP32 force passes read fractions)
    if (cells) {
        const size_t C = (size_t)S.ncells;
        S.want(&S.xa, v4 * N);
        S.want(&S.xcs, v4 * N);
        S.want(&S.q, sizeof(int4) * N);
        S.want(&S.cell_of, sizeof(int) * N);
        S.want(&S.perm, sizeof(int) * N);
        S.want(&S.cell_start, sizeof(int) * (C + 1));
        S.want(&S.cell_count, sizeof(int) * C);
        S.want(&S.cell_cursor, sizeof(int) * C);
        S.want(&S.scan_sums, sizeof(int) * 1024);
    }
}

int commit1(Scratch1& S, int n, const double box[3], double rcs, const int n3[3], int prec,
            const nefe_sw_params* prm, const nefe_uf_params* uf, double skin) {
    const int ntiles = (n + kTile - 1) / kTile;
    DevSys hs;
    std::memset(&hs, 0, sizeof(hs));
    hs.off = 0; hs.n = n; hs.tile0 = 0; hs.ntile = ntiles; hs.cell0 = 0;
    hs.ncell_cap = n3[0] * n3[1] * n3[2];
    hs.rcs = rcs; hs.pair = -1; hs.prm = 0; hs.mass_e = 1.0;
    hs.rcs2_lo_f = (float)(rcs * rcs) * (1.0f - 1e-4f);
    hs.rcs2_hi_f = (float)(rcs * rcs) * (1.0f + 1e-4f);
    if (uf) {
        fill_uf(hs, *uf, skin, UF_INT);
        hs.pot = POT_UF;
    }
    DevState st;
    std::memset(&st, 0, sizeof(st));
    set_grid(st, box, n3);
    st.rebuild = 1;
    st.scale_int = 1.0;
    SwcBytes sw;
    std::memset(&sw, 0, sizeof(sw));
    if (prm && prec == NEFE_FP32) {
        const SWc<float> c = make_swc<float>(*prm);
        std::memcpy(sw.b, &c, sizeof(c));
        hs.leg_unit_f = 1.0f / c.leg_scale;
    }
    NEFE_CU(S.commit());
    const int nacc = 2 * ACC_N * kSlots;
    const int work = std::max(std::max(ntiles, S.ncells), nacc);
    k_scratch_init<<<std::min((work + 255) / 256, 608), 256, 0, S.s>>>(
        hs, st, sw, S.sys, S.st, S.swc, S.tiles, ntiles, S.acc, nacc, S.cell_count, S.ncells);
    NEFE_CU(cudaGetLastError());
    return NEFE_OK;
}

Bufs bufs_of(const Scratch1& S, const double* x, int n) {
    Bufs b;
    std::memset(&b, 0, sizeof(b));
    b.sys = S.sys; b.st = S.st; b.acc = S.acc; b.acc_lo = S.acc + ACC_N * kSlots; b.tiles = S.tiles;
    b.x = const_cast<double*>(x);
    b.xs = S.xs; b.xa = S.xa; b.xcs = S.xcs; b.q = S.q; b.cell_of = S.cell_of; b.perm = S.perm;
    b.shd = S.shd; b.shj = S.shj; b.shn = S.shn; b.P = S.P;
    b.cell_start = S.cell_start; b.cell_count = S.cell_count; b.cell_cursor = S.cell_cursor;
    b.ntot = n; b.swc = S.swc;
    b.scan_sums = S.scan_sums; b.ncells_host = S.ncells;
    return b;
}

}  // namespace nefe

using namespace nefe;

// The call's error word, after its work on the stream.
static int read_error(const Scratch1& S, unsigned* err) {
    NEFE_CU(cudaMemcpyAsync(err, &S.st->err, sizeof(*err), cudaMemcpyDeviceToHost, S.s));
    NEFE_CU(cudaStreamSynchronize(S.s));
    return NEFE_OK;
}

// Scratch of the two force passes: the scatter form's accumulators (FP32), or the shells, leg
// forces and partial forces of the gather form (FP64).
static void want_forces(Scratch1& S, int n, int precision) {
    const size_t N = (size_t)n;
    S.want(&S.shn, sizeof(int) * N);
    S.want(&S.xc, sizeof(uint2) * N);
    S.want(&S.lscale, sizeof(float4) * 4);
    if (precision == NEFE_FP32) {
        S.want(&S.xf, sizeof(int4) * N);
        S.want(&S.lacc, 4 * sizeof(int) * N);
        S.want(&S.lacc_hi, 3 * sizeof(long long) * N);
        S.want(&S.hi_flag, sizeof(int) * ((N + kTile - 1) / kTile));
    } else {
        S.want(&S.shd, sizeof(double4) * N * kShell);
        S.want(&S.shj, sizeof(int) * N * kShell);
        S.want(&S.P, sizeof(double4) * N);
    }
}

// Both force passes of a stateless call.  FP64 pass B: one lane per atom from kGatherOne atoms on (its
// epilogue runs on one lane per atom, so more lanes cost FP64 issue; fewer atoms want shorter chains).
constexpr int kGatherOne = 20000;
static int run_forces(const Scratch1& S, Bufs& b, int n, const double box[3], const nefe_sw_params* prm, int precision) {
    const int ntiles = (n + kTile - 1) / kTile;
    b.xc = S.xc; b.lscale = S.lscale;
    b.row4 = (b.cap & 3) == 0 && (reinterpret_cast<uintptr_t>(b.nbr) & 15) == 0;
    set_edge_items(b, precision, atoms_per_warp_log2(precision, n), ntiles);
    b.common = 1;
    if (precision == NEFE_FP32) {
        b.xf = S.xf; b.want_xf = 1 + frac_fine(box); b.lacc = S.lacc; b.lacc_hi = S.lacc_hi; b.hi_flag = S.hi_flag;
        b.swc_common = make_swc<float>(*prm);
        NEFE_CU(cudaMemsetAsync(S.lacc, 0, (size_t)(reinterpret_cast<char*>(S.hi_flag + ntiles) - reinterpret_cast<char*>(S.lacc)),
                                S.s));
        launch_frac_positions(b, S.s);
        launch_edges(b, precision, 0, ntiles, FM_FORCES, S.s, nullptr);
        launch_gather(b, precision, 0, ntiles, FM_FORCES, S.s, nullptr);
    } else {
        b.swp_common = sw_params_real(*prm);
        launch_mirror(b, precision, ntiles, S.s, nullptr);
        launch_edges(b, precision, 8, ntiles, FM_FORCES, S.s, nullptr);
        launch_gather(b, precision, n >= kGatherOne ? 1 : 4, ntiles, FM_FORCES, S.s, nullptr);
    }
    NEFE_CU(cudaGetLastError());
    return NEFE_OK;
}

extern "C" {

const char* nefe_last_error(void) { return g_msg; }

int nefe_sw_params_silicon(nefe_sw_params* out) {
    if (!out) return fail(NEFE_EINVAL, "out is NULL");
    out->eps = 2.1683; out->sigma = 2.0951; out->A = 7.049556277; out->B = 0.6022245584;
    out->p = 4.0; out->q = 0.0; out->a = 1.80; out->lambda3 = 21.0; out->gamma = 1.20;
    out->cos0 = -1.0 / 3.0;
    return NEFE_OK;
}

int nefe_cell_bin(const double* x, int n, const double box[3], double rcs, int ncell3[3],
                  int* cell_of, int* cell_start, int* perm, int ncell_cap, void* stream) {
    NvtxRange nvtx_("nefe_cell_bin");
    if (n < 0 || !box || !ncell3 || (n > 0 && (!x || !cell_of || !perm)) || !cell_start)
        return fail(NEFE_EINVAL, "nefe_cell_bin: bad argument");
    if (n >= (1 << kCodeShift)) return fail(NEFE_EINVAL, "nefe_cell_bin: n above 2^27");
    int rc = check_box(box, rcs);
    if (rc) return rc;
    int n3[3];
    if (!host_grid(box, rcs, n3)) return fail(NEFE_EINVAL, "nefe_cell_bin: fewer than 2 cells on an axis");
    const long long total = (long long)n3[0] * n3[1] * n3[2];
    if (total > ncell_cap) return fail(NEFE_EINVAL, "nefe_cell_bin: %lld cells above capacity %d", total, ncell_cap);
    for (int k = 0; k < 3; ++k) ncell3[k] = n3[k];
    Scratch1 S;
    S.s = (cudaStream_t)stream;
    if (n == 0) {
        NEFE_CU(cudaMemsetAsync(cell_start, 0, sizeof(int) * (size_t)(total + 1), S.s));
        return NEFE_OK;
    }
    want1(S, n, n3, NEFE_FP32, true);
    rc = commit1(S, n, box, rcs, n3, NEFE_FP32);
    if (rc) return rc;
    Bufs b = bufs_of(S, x, n);
    b.cell_of = cell_of; b.perm = perm; b.cell_start = cell_start;
    launch_cells(b, NEFE_FP32, (n + kTile - 1) / kTile, 1, 1, S.s, nullptr);
    launch_cells_sort(b, (int)total, S.s);
    NEFE_CU(cudaGetLastError());
    return NEFE_OK;
}

int nefe_neighbor_build(const double* x, int n, const double box[3], double rcs, int cap,
                        int* nbr, int* cnt, int* overflow, void* stream) {
    NvtxRange nvtx_("nefe_neighbor_build");
    if (n < 0 || !box || cap < 1 || cap > kMaxCap || (n > 0 && (!x || !nbr || !cnt)))
        return fail(NEFE_EINVAL, "nefe_neighbor_build: bad argument");
    if (n >= (1 << kCodeShift)) return fail(NEFE_EINVAL, "nefe_neighbor_build: n above 2^27");
    int rc = check_box(box, rcs);
    if (rc) return rc;
    if (overflow) *overflow = 0;
    if (n == 0) return NEFE_OK;
    int n3[3];
    if (!host_grid(box, rcs, n3)) return fail(NEFE_EINVAL, "nefe_neighbor_build: fewer than 2 cells on an axis");
    const long long total = (long long)n3[0] * n3[1] * n3[2];
    if (total > (1LL << 30)) return fail(NEFE_EINVAL, "nefe_neighbor_build: cell grid too large");
    Scratch1 S;
    S.s = (cudaStream_t)stream;
    want1(S, n, n3, NEFE_FP32, true);
    rc = commit1(S, n, box, rcs, n3, NEFE_FP32);
    if (rc) return rc;
    Bufs b = bufs_of(S, x, n);
    b.nbr = nbr; b.cnt = cnt; b.cap = cap;
    launch_cells_and_list(b, NEFE_FP32, (n + kTile - 1) / kTile, 1, 1, S.s, nullptr);
    NEFE_CU(cudaGetLastError());
    unsigned err = 0;
    if ((rc = read_error(S, &err))) return rc;
    const int ovf = (err & NEFE_ERR_NBR_OVERFLOW) ? 1 : 0;
    if (overflow) *overflow = ovf;
    if (ovf) return fail(NEFE_EOVERFLOW, "nefe_neighbor_build: a row exceeded cap %d", cap);
    return NEFE_OK;
}

int nefe_sw_forces(const double* x, int n, const double box[3], double rcs, const int* nbr,
                   const int* cnt, int cap, const nefe_sw_params* prm, int precision, double* f,
                   double* e_atom, double* energy_virial, int* shell_overflow, void* stream) {
    NvtxRange nvtx_("nefe_sw_forces");
    if (n < 0 || !box || cap < 1 || cap > kMaxCap || !valid_params(prm) ||
        (precision != NEFE_FP32 && precision != NEFE_FP64) || (n > 0 && (!x || !nbr || !cnt || !f)))
        return fail(NEFE_EINVAL, "nefe_sw_forces: bad argument");
    if (prm->a * prm->sigma > rcs) return fail(NEFE_EINVAL, "nefe_sw_forces: a*sigma above rcs");
    int rc = check_box(box, rcs);
    if (rc) return rc;
    if (shell_overflow) *shell_overflow = 0;
    int n3[3];
    if (!host_grid(box, rcs, n3)) return fail(NEFE_EINVAL, "nefe_sw_forces: fewer than 2 cells on an axis");
    cap_grid(n3, 1LL << 30);
    Scratch1 S;
    S.s = (cudaStream_t)stream;
    want1(S, n, n3, precision, false);
    want_forces(S, n, precision);
    if ((rc = commit1(S, n, box, rcs, n3, precision, prm))) return rc;
    if (n > 0) {
        Bufs b = bufs_of(S, x, n);
        b.nbr = const_cast<int*>(nbr); b.cnt = const_cast<int*>(cnt); b.cap = cap;
        b.f_out = f; b.e_atom = e_atom;
        if ((rc = run_forces(S, b, n, box, prm, precision))) return rc;
    }
    if (energy_virial) launch_decode_ev(S.acc, energy_virial, &S.st->err, S.s);
    NEFE_CU(cudaGetLastError());
    if (shell_overflow) {
        unsigned err = 0;
        if ((rc = read_error(S, &err))) return rc;
        *shell_overflow = (err & NEFE_ERR_SHELL_OVERFLOW) ? 1 : 0;
        if (*shell_overflow) return fail(NEFE_EOVERFLOW, "nefe_sw_forces: shell above 32 neighbours");
    }
    return NEFE_OK;
}

int nefe_sw_energy_grad(const double* x, int n, const double box[3], double rcs, const int* nbr,
                        const int* cnt, int cap, const nefe_sw_params* prm, int precision, double* f,
                        double* energy_grad, void* stream) {
    NvtxRange nvtx_("nefe_sw_energy_grad");
    if (n < 0 || !box || cap < 1 || cap > kMaxCap || !valid_params(prm) || !energy_grad ||
        (precision != NEFE_FP32 && precision != NEFE_FP64) || (n > 0 && (!x || !nbr || !cnt)))
        return fail(NEFE_EINVAL, "nefe_sw_energy_grad: bad argument");
    if (prm->a * prm->sigma > rcs) return fail(NEFE_EINVAL, "nefe_sw_energy_grad: a*sigma above rcs");
    int rc = check_box(box, rcs);
    if (rc) return rc;
    int n3[3];
    if (!host_grid(box, rcs, n3)) return fail(NEFE_EINVAL, "nefe_sw_energy_grad: fewer than 2 cells on an axis");
    cap_grid(n3, 1LL << 30);
    Scratch1 S;
    S.s = (cudaStream_t)stream;
    want1(S, n, n3, precision, false);
    double* fo = f;
    if (!fo) S.want(&fo, sizeof(double) * 3 * (size_t)n);
    want_forces(S, n, precision);
    if ((rc = commit1(S, n, box, rcs, n3, precision, prm))) return rc;
    if (n > 0) {
        Bufs b = bufs_of(S, x, n);
        b.nbr = const_cast<int*>(nbr); b.cnt = const_cast<int*>(cnt); b.cap = cap;
        b.f_out = fo; b.e_atom = nullptr; b.want_grad = 1;
        if ((rc = run_forces(S, b, n, box, prm, precision))) return rc;
    }
    launch_decode_grad(S.acc, energy_grad, S.s);
    NEFE_CU(cudaGetLastError());
    unsigned err = 0;
    if ((rc = read_error(S, &err))) return rc;
    if (err & NEFE_ERR_SHELL_OVERFLOW)
        return fail(NEFE_EOVERFLOW, "nefe_sw_energy_grad: shell above 32 neighbours");
    if (err & NEFE_ERR_NAN) return fail(NEFE_ENAN, "nefe_sw_energy_grad: non-finite sum");
    return NEFE_OK;
}

int nefe_uf_forces(const double* x, int n, const double box[3], double rcs, double skin,
                   const nefe_uf_params* uf, int precision, double* f, double* e_atom,
                   double* energy_virial, void* stream) {
    NvtxRange nvtx_("nefe_uf_forces");
    if (n < 0 || !box || !valid_uf(uf) || !(skin >= 0.0) || (precision != NEFE_FP32 && precision != NEFE_FP64) ||
        (n > 0 && (!x || !f)))
        return fail(NEFE_EINVAL, "nefe_uf_forces: bad argument");
    if (n >= (1 << kUfShift)) return fail(NEFE_EINVAL, "nefe_uf_forces: n above 2^25");
    int rc = check_box(box, rcs);
    if (rc) return rc;
    const double R = uf->rc + skin;
    if (R > 2.0 * rcs) return fail(NEFE_EINVAL, "nefe_uf_forces: rc + skin = %g above 2 rcs = %g", R, 2.0 * rcs);
    int n3[3];
    if (!host_grid(box, rcs, n3)) return fail(NEFE_EINVAL, "nefe_uf_forces: fewer than 2 cells on an axis");
    for (int k = 0; k < 3; ++k) {
        if (n3[k] < 5) return fail(NEFE_EINVAL, "nefe_uf_forces: fewer than 5 cells on an axis");
        if (box[k] < 2.0 * R) return fail(NEFE_EINVAL, "nefe_uf_forces: box below 2 (rc + skin)");
    }
    const long long total = (long long)n3[0] * n3[1] * n3[2];
    if (total > (1LL << 30)) return fail(NEFE_EINVAL, "nefe_uf_forces: cell grid too large");
    Scratch1 S;
    S.s = (cudaStream_t)stream;
    want1(S, n, n3, precision, true);
    int* uf_nbr = nullptr;
    int* uf_cnt = nullptr;
    S.want(&uf_nbr, sizeof(int) * (size_t)n * kUfCap);
    S.want(&uf_cnt, sizeof(int) * (size_t)n);
    if (precision == NEFE_FP32) {
        S.want(&S.xf, sizeof(int4) * (size_t)n);
        S.want(&S.xc, sizeof(uint2) * (size_t)n);
        S.want(&S.lscale, sizeof(float4) * 4);
    }
    if ((rc = commit1(S, n, box, rcs, n3, precision, nullptr, uf, skin))) return rc;
    if (n > 0) {
        Bufs b = bufs_of(S, x, n);
        b.uf_nbr = uf_nbr; b.uf_cnt = uf_cnt; b.uf_tiles = nullptr;
        b.xf = b.xfb = S.xf; b.xc = S.xc; b.lscale = S.lscale;
        b.want_xf = precision == NEFE_FP32 ? 1 + frac_fine(box) : 0;
        b.f_out = f; b.e_atom = e_atom;
        const int ntiles = (n + kTile - 1) / kTile;
        launch_cells(b, precision, ntiles, 1, 1, S.s, nullptr);
        launch_uf_list(b, precision, ntiles, 1, 1, S.s, nullptr);
        launch_uf(b, precision, ntiles, FM_FORCES, S.s, nullptr);
        NEFE_CU(cudaGetLastError());
    }
    if (energy_virial) launch_decode_ev(S.acc, energy_virial, nullptr, S.s);
    NEFE_CU(cudaGetLastError());
    unsigned err = 0;
    if ((rc = read_error(S, &err))) return rc;
    if (err & NEFE_ERR_NBR_OVERFLOW) return fail(NEFE_EOVERFLOW, "nefe_uf_forces: a row exceeded %d", kUfCap);
    if (err & (NEFE_ERR_BOX | NEFE_ERR_CELL)) return fail(NEFE_EINVAL, "nefe_uf_forces: cell grid error");
    return NEFE_OK;
}

int nefe_release_scratch(void) {
    NvtxRange nvtx_("nefe_release_scratch");
    NEFE_CU(scratch_release());
    return NEFE_OK;
}

int nefe_check_barrier_timeout(int device, double limit_ms) {
    if (!(limit_ms > 0.0 && limit_ms <= 1000.0)) return fail(NEFE_EINVAL, "limit_ms must be in (0, 1000]");
    NEFE_CU(cudaSetDevice(device));
    const int r = check_barrier_timeout(limit_ms);
    if (r < 0) return fail(NEFE_ECUDA, "barrier check: CUDA error");
    return r ? fail(NEFE_ETIMEOUT, "the barrier gave up by its limit (expected)") : NEFE_OK;
}

int nefe_langevin_noise(uint64_t seed, uint64_t sys_id, uint64_t step, int n, int precision,
                        double* xi, void* stream) {
    NvtxRange nvtx_("nefe_langevin_noise");
    if (n < 0 || (n > 0 && !xi) || (precision != NEFE_FP32 && precision != NEFE_FP64))
        return fail(NEFE_EINVAL, "nefe_langevin_noise: bad argument");
    launch_noise(seed, sys_id, step, n, precision, xi, (cudaStream_t)stream);
    NEFE_CU(cudaGetLastError());
    return NEFE_OK;
}

}  // extern "C"
