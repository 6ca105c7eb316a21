// libnefe device kernels for sm_103a.
//
// Step sequence of one time step k -> k+1 (all systems of a context at once):
//   k_group       per system / dCCI pair: reads the fixed-point sums of step k, observes
//                 P, V, dH/dl, records, kicks the barostat, advances lambda and W (Eq. Wdyn,
//                 left point), applies the dCCI update (Eqs. Ps_coex_discreted /
//                 l_coex_discreted), sets this step's drift factors and zeroes the sums.
//   k_kick_drift  v += dt/2 F/m; displacement since the last list build += dt phi v (+ the
//                 affine box drift), kept as a compensated pair in the FP32 path; position as
//                 the force pass in use reads it (fractions of the box, packed fractions for the
//                 row filter, mirror xs = x - q h); displacement test -> rebuild flag;
//                 thermostat noise + its sum.
//                 In the scatter form this work is done by the previous step's epilogue for the
//                 systems without a barostat (k_finish with fuse), and the kernel skips them.
//   rebuild       (flagged systems) fold the displacement into the FP64 anchor, cell count ->
//                 scan -> fill (with a cell-ordered copy of the mirror) -> Verlet list: a cluster
//                 of blocks per system up to the fill (k_cells_clusters, few small systems), or a
//                 kernel sequence over a worklist, or one cooperative launch (k_rebuild_coop).
//                 Uhlenbeck-Ford rows (k_uflist) by the same cells.
//   k_edges_s     force pass A of the scatter form (the FP32 default): the edges of a warp's atoms
//                 as one list, pair terms, the shells' moments and the force each atom's terms
//                 exert on each leg atom, added into int32 fixed-point accumulators (order
//                 independent).  k_edges1, k_edges: the FP32 gather form with one thread or a
//                 lane group per atom, storing per edge.  k_edges_d: FP64, edge lists of a warp's
//                 atoms, storing per edge.  k_uf: Uhlenbeck-Ford forces, several lanes per atom.
//   k_finish      the scatter form's epilogue: reads and clears the accumulators; Einstein
//                 springs, lambda mixing, Langevin force with its per-system mean removed,
//                 second half kick (and the next step's kick, drift and noise, see above).
//   k_gather      force pass B of the gather form: the atom's pass-A force plus the leg forces
//                 that the triplets centred on its neighbours exert on it, then the same
//                 epilogue.
//
// Positions: the FP64 anchor x (positions at the last list build) plus the displacement
// since then (FP64, or an FP32 value + FP32 compensation term, ~2^-48 relative).  The anchor
// absorbs the displacement at every list build, so the per-step path of the FP32 kernels
// issues no FP64 instruction (GB300 runs FP64 at 1/64 of the FP32 rate): per-system
// constants are read from FP32 copies written once per step by k_group.
#include <cuda_runtime.h>
#include <stdint.h>

#include "nefe.h"
#include "nefe_dev.h"
#include "nefe_launch.h"
#include "nefe_sw_terms.h"

namespace nefe {

// Every kernel here waits, before its first memory access, for the launch before it to have completed
// (dep_wait; a kernel that does not use its result waits as well, so that completion stays transitive
// along the stream), and is launched with programmatic stream serialization: its blocks are then
// resident already when the last block before them ends.  A step is 8 to 10 dependent launches of a
// few us each, and what this takes off is the start of each.  One 8000-atom FP32 system
// 28.3 -> 26.0 us a step, 64 atoms in FP64 50.8 -> 48.0 us.  Not after a long launch that fills the chip: the blocks would
// go to the SMs that finish first and leave the others idle (16 x 8000 atoms in FP64: gather 57 -> 90 us), so
// the kernels that follow the pair passes use it up to kEarlyBlocks blocks only, and the group update
// up to kEarlyGroups.  Launched without the attribute the two instructions do nothing.
constexpr int kEarlyBlocks = 2 * 152, kEarlyGroups = 32;
__device__ __forceinline__ void dep_wait() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
template <typename T> struct Same { using t = T; };
template <typename... P>
static void launch_next_if(bool early, void (*kernel)(P...), int blocks, int threads, cudaStream_t s, typename Same<P>::t... args) {
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3((unsigned)threads);
    cfg.stream = s;
    cudaLaunchAttribute attr{};
    attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &attr;
    cfg.numAttrs = early ? 1 : 0;
    cudaLaunchKernelEx(&cfg, kernel, args...);
}
template <typename... P>
static void launch_next(void (*kernel)(P...), int blocks, int threads, cudaStream_t s, typename Same<P>::t... args) {
    launch_next_if(true, kernel, blocks, threads, s, args...);
}

template <typename T> struct V4;
template <> struct V4<float> { using t = float4; };
template <> struct V4<double> { using t = double4; };

__device__ __forceinline__ float4 mk4(float a, float b, float c, float d) { return make_float4(a, b, c, d); }
__device__ __forceinline__ double4 mk4(double a, double b, double c, double d) { return make_double4(a, b, c, d); }

// Precision-explicit math (no silent promotion of FP32 arguments to the FP64 routines).
// The FP32 path uses the hardware approximations (MUFU: ex2, rcp, rsqrt; a few ulp, far
// inside the 1e-5 relative force tolerance); the FP64 path the correctly rounded routines.
__device__ __forceinline__ float xexp(float v) { return __expf(v); }
__device__ __forceinline__ double xexp(double v) { return ::exp(v); }
__device__ __forceinline__ float xrcp(float v) { return __fdividef(1.0f, v); }
__device__ __forceinline__ double xrcp(double v) { return 1.0 / v; }
__device__ __forceinline__ float xrsqrt(float v) { return rsqrtf(v); }
__device__ __forceinline__ double xrsqrt(double v) { return ::rsqrt(v); }
__device__ __forceinline__ float xpow(float a, float b) { return __powf(a, b); }
__device__ __forceinline__ float xlog(float v) { return __logf(v); }
__device__ __forceinline__ double xlog(double v) { return ::log(v); }
__device__ __forceinline__ double xpow(double a, double b) { return ::pow(a, b); }

// FP32 copy or FP64 source of a constant, by kernel precision.
template <typename T> __device__ __forceinline__ T pick(double d, float f) {
    if constexpr (sizeof(T) == 4) return f; else return d;
}

// ------------------------------------------------------------------------------------
// Philox4x64-10 (Salmon, Moraes, Dror, Shaw, SC'11): round (hi0,lo0) = M0 X0,
// (hi1,lo1) = M1 X2, X <- (hi1^X1^k0, lo1, hi0^X3^k1, lo0), key += Weyl constants.
// ------------------------------------------------------------------------------------
__device__ __forceinline__ void philox4x64_10(uint64_t c[4], uint64_t k0, uint64_t k1) {
    const uint64_t M0 = 0xD2E7470EE14C6C93ULL, M1 = 0xCA5A826395121157ULL;
    const uint64_t W0 = 0x9E3779B97F4A7C15ULL, W1 = 0xBB67AE8584CAA73BULL;
#pragma unroll
    for (int r = 0; r < 10; ++r) {
        const uint64_t hi0 = __umul64hi(M0, c[0]), lo0 = M0 * c[0];
        const uint64_t hi1 = __umul64hi(M1, c[2]), lo1 = M1 * c[2];
        const uint64_t n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
        c[0] = n0; c[1] = lo1; c[2] = n2; c[3] = lo0;
        k0 += W0; k1 += W1;
    }
}

// Three standard normals for (seed, system, step, atom): counter (step, atom, system, 0),
// key (seed, 0); Box-Muller on the (0,1) uniforms of outputs (0,1) and (2,3).
template <typename T> struct Noise;
template <> struct Noise<double> {
    __device__ static void xi3(uint64_t seed, uint64_t sys, uint64_t step, uint64_t id, double out[3]) {
        uint64_t c[4] = {step, id, sys, 0ULL};
        philox4x64_10(c, seed, 0ULL);
        double unused;
        pair(c[0], c[1], out[0], out[1]);
        pair(c[2], c[3], out[2], unused);
    }
    // Box-Muller pair of two words
    __device__ __forceinline__ static void pair(uint64_t c0, uint64_t c1, double& a, double& b) {
        const double u0 = ((double)(c0 >> 11) + 0.5) * 0x1p-53, u1 = ((double)(c1 >> 11) + 0.5) * 0x1p-53;
        const double r = ::sqrt(__dmul_rn(-2.0, ::log(u0)));
        double sn, cs;
        ::sincospi(2.0 * u1, &sn, &cs);
        a = __dmul_rn(r, cs);
        b = __dmul_rn(r, sn);
    }
};
template <> struct Noise<float> {
    __device__ static void xi3(uint64_t seed, uint64_t sys, uint64_t step, uint64_t id, float out[3]) {
        uint64_t c[4] = {step, id, sys, 0ULL};
        philox4x64_10(c, seed, 0ULL);
        const float u0 = ((float)(uint32_t)(c[0] >> 40) + 0.5f) * 0x1p-24f;
        const float u1 = ((float)(uint32_t)(c[1] >> 40) + 0.5f) * 0x1p-24f;
        const float u2 = ((float)(uint32_t)(c[2] >> 40) + 0.5f) * 0x1p-24f;
        const float u3 = ((float)(uint32_t)(c[3] >> 40) + 0.5f) * 0x1p-24f;
        const float r0 = sqrtf(-2.0f * logf(u0)), r1 = sqrtf(-2.0f * logf(u2));
        float s0, c0, s1, c1;
        sincospif(2.0f * u1, &s0, &c0);
        sincospif(2.0f * u3, &s1, &c1);
        out[0] = r0 * c0; out[1] = r0 * s0; out[2] = r1 * c1;
    }
};

// ------------------------------------------------------------------------------------
// Deterministic per-system sums: warp shuffle in kernel precision, then the block's warp
// partials summed in kernel precision in a fixed order, then one int64 fixed-point atomic per
// value into slot (blockIdx % kSlots).  The FP64 path converts the block sum at 2^-32; the
// FP32 path rounds it to a multiple of 2^-16 (an int32 conversion, |block sum| < 32768) before
// moving it to the 2^-32 scale, so a block's contribution carries at most 2^-17 of rounding
// on top of its FP32 summation error.  A larger block sum is converted warp by warp: what cannot be
// summed (and is reported) are 32,768 eV in a warp (32 atoms at most; 65,536 for dE/dtheta), whatever
// the block's size.  Integer addition makes the per-system total independent of the order in which
// blocks arrive.  Every thread of the block must call it.
// In FP64 the threads' values are converted first (2^-40 units) and summed as integers: FP64 adds
// run at 2 lanes a cycle, and five of them per value and warp were a third of the epilogue.  The
// integer sum of a block (at most 128 threads) stays below 2^62 when every value is below 2^15; a
// block that holds a larger value (or one that is not finite) takes the FP64 sums.  The remainders of
// the conversion to 2^-32 are kept in slots of their own (acc_lo) where blocks are small: 8 atoms to a
// block round four times as often as 32.
// ------------------------------------------------------------------------------------
// Rows of the remainders of pass A's sums (U_int, virial).  The engine keeps them in the rows of
// dE/dtheta, which it has no other use for (and which its saved states hold); the stateless calls have
// a second array of the sums' layout.
__device__ __forceinline__ int engine_lo_row(int a) { return ACC_DTH + max(a - 1, 0); }

template <typename T, int K>
__device__ __forceinline__ void block_sum_to_acc(T (&v)[K], long long* acc_sys, int first,
                                                 unsigned* err, long long* acc_lo = nullptr,
                                                 bool engine = false) {
    if constexpr (sizeof(T) == 8) {
        __shared__ long long ired[kTile / 32][K];
        constexpr double most = 4194304.0 / kTile;
        bool big = false;
#pragma unroll
        for (int k = 0; k < K; ++k) big = big || !(fabs(v[k]) < most);
        if (!__syncthreads_or(big)) {
            const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
            for (int k = 0; k < K; ++k) {
                long long q = __double2ll_rn(v[k] * 0x1p40);
#pragma unroll
                for (int o = 16; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
                if (lane == 0) ired[w][k] = q;
            }
            __syncthreads();
            if (threadIdx.x < K) {
                long long s = 0;
                for (int i = 0; i < (int)(blockDim.x >> 5); ++i) s += ired[i][threadIdx.x];
                const int a = first + (int)threadIdx.x, slot = (int)(blockIdx.x % kSlots);
                const long long units = s;
                s = (s + 128) >> 8;
                if (s != 0)
                    atomicAdd(reinterpret_cast<unsigned long long*>(&acc_sys[a * kSlots + slot]), (unsigned long long)s);
                if (acc_lo && units != s * 256)
                    atomicAdd(reinterpret_cast<unsigned long long*>(&acc_lo[(engine ? engine_lo_row(a) : a) * kSlots + slot]),
                              (unsigned long long)(units - s * 256));
            }
            return;
        }
    }
    __shared__ T red[kTile / 32][K];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < K; ++k) {
        T x = v[k];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane == 0) red[w][k] = x;
    }
    __syncthreads();
    if (threadIdx.x < K) {
        T s = 0;
        const int nw = (int)(blockDim.x >> 5);
        for (int i = 0; i < nw; ++i) s += red[i][threadIdx.x];
        long long q;
        bool bad;
        if constexpr (sizeof(T) == 4) {
            // round(s 2^16) in int32 (|s| < 32768 per block), moved to the 2^-32 scale
            const float t = s * 65536.0f;
            bad = !(fabsf(t) < 2147483520.0f);
            q = bad ? 0LL : (long long)__float2int_rn(t) * 65536LL;
            if (bad) {                           // rare: the warps' sums one by one
                constexpr float most = K == 7 ? 4294967040.0f : 2147483520.0f;   // (K = 7: dE/dtheta)
                bad = false;
                for (int i = 0; i < nw; ++i) {
                    const float u = red[i][threadIdx.x] * 65536.0f;
                    if (fabsf(u) < most) q += __float2ll_rn(u) * 65536LL;
                    else bad = true;
                }
            }
        } else {
            bad = !isfinite(s);
            q = bad ? 0LL : __double2ll_rn(s * kFix);
        }
        if (bad) {
            atomicOr(err, NEFE_ERR_NAN);
        } else if (q != 0) {
            atomicAdd(reinterpret_cast<unsigned long long*>(
                          &acc_sys[(size_t)(first + threadIdx.x) * kSlots + (blockIdx.x % kSlots)]),
                      (unsigned long long)q);
        }
    }
}

// Sum of the kSlots fixed-point slots of one per-system value.  The loads are independent, so
// they are issued together (one memory latency, not kSlots of them).
__device__ __forceinline__ long long slot_sum(const long long* slots) {
    long long v[kSlots];
#pragma unroll
    for (int sl = 0; sl < kSlots; ++sl) v[sl] = slots[sl];
    long long sum = 0;
#pragma unroll
    for (int sl = 0; sl < kSlots; ++sl) sum += v[sl];
    return sum;
}

// Per-block table of the 27 cell-offset vectors o h (o in {-1,0,1}^3), indexed by the list
// entry's code.  Every thread of the block must call it.
template <typename T>
__device__ __forceinline__ void offset_table(typename V4<T>::t* tab, T hx, T hy, T hz) {
    if (threadIdx.x < 27) {
        const int c = threadIdx.x;
        const int ox = c % 3 - 1, oy = (c / 3) % 3 - 1, oz = c / 9 - 1;
        tab[c] = mk4(ox == 0 ? (T)0 : (ox < 0 ? -hx : hx), oy == 0 ? (T)0 : (oy < 0 ? -hy : hy),
                     oz == 0 ? (T)0 : (oz < 0 ? -hz : hz), (T)0);
    }
    __syncthreads();
}

// The same 27 offset vectors as three component rows of 32 (row k, entry c at tab[32 k + c]):
// a warp whose lanes index different entries reads each row without bank conflicts (a table
// of 16-byte vectors indexed at random serialises).  Every thread of the block must call it.
template <typename T>
__device__ __forceinline__ void offset_rows(T* tab, T hx, T hy, T hz) {
    if (threadIdx.x < 27) {
        const int c = threadIdx.x;
        const int ox = c % 3 - 1, oy = (c / 3) % 3 - 1, oz = c / 9 - 1;
        tab[c] = ox == 0 ? (T)0 : (ox < 0 ? -hx : hx);
        tab[32 + c] = oy == 0 ? (T)0 : (oy < 0 ? -hy : hy);
        tab[64 + c] = oz == 0 ? (T)0 : (oz < 0 ? -hz : hz);
    }
    __syncthreads();
}

// Cell grid for a box: per axis floor(L/rcs), reduced while L/n < rcs (1 + 1e-9); then the
// largest axis is reduced until the product fits the capacity (wider cells stay valid).
__device__ __forceinline__ bool grid_for(const double box[3], double rcs, int cap, int n3[3]) {
    bool ok = true;
    for (int k = 0; k < 3; ++k) {
        int m = (int)floor(__ddiv_rn(box[k], rcs));
        while (m > 0 && __ddiv_rn(box[k], (double)m) < rcs * (1.0 + 1e-9)) --m;
        if (m < 2) { ok = false; m = 2; }
        n3[k] = m;
    }
    while ((long long)n3[0] * n3[1] * n3[2] > cap) {
        int k = (n3[0] >= n3[1] && n3[0] >= n3[2]) ? 0 : (n3[1] >= n3[2] ? 1 : 2);
        if (n3[k] <= 2) { ok = false; break; }
        --n3[k];
    }
    return ok;
}

// FP32 copies of the box-dependent constants (called wherever h or hb change).
__device__ __forceinline__ void refresh_box_f(DevState& st) {
    bool hm = false;
    for (int k = 0; k < 3; ++k) {
        st.h_f[k] = (float)st.h[k];
        st.hb_f[k] = (float)st.hb[k];
        st.rho_f[k] = (float)(st.h[k] / st.hb[k]);
        hm = hm || (st.h[k] != st.hb[k]);
    }
    st.hmoved = hm ? 1 : 0;
}

struct TileAtom {
    int sys, first, count;
};
// One load: the kernels' first operands wait for it, so the system descriptor is not in their way.
__device__ __forceinline__ TileAtom tile_of(const Bufs& b, int tile) {
    const int4 v = b.tiles[tile];
    TileAtom t;
    t.sys = v.x;
    t.first = v.y;
    t.count = v.z;
    return t;
}

// A tile's system descriptor and state copied into shared memory by all threads of the block
// (independent 4-byte loads: one memory latency, instead of one per cache line of the structs
// that the kernel's field accesses would otherwise wait for, one after the other).  Writes to the
// state (flags, error bits) still go to the global copy.  The caller syncs.
struct StagedSys {
    DevSys S;
    DevState st;
};
__device__ __forceinline__ void stage_sys(const Bufs& b, int sys, StagedSys& sh) {
    const uint32_t* gs = reinterpret_cast<const uint32_t*>(b.sys + sys);
    const uint32_t* gt = reinterpret_cast<const uint32_t*>(b.st + sys);
    uint32_t* ds = reinterpret_cast<uint32_t*>(&sh.S);
    uint32_t* dt = reinterpret_cast<uint32_t*>(&sh.st);
    constexpr int ws = (int)(sizeof(DevSys) / 4), wt = (int)(sizeof(DevState) / 4);
    for (int w = threadIdx.x; w < ws + wt; w += blockDim.x) {
        if (w < ws) ds[w] = gs[w];
        else dt[w - ws] = gt[w - ws];
    }
}

// ------------------------------------------------------------------------------------
// Cell of a coordinate along one axis: the unwrapped cell index q = floor(x/L) n + c and the cell
// c in [0, n), with c = (int)(w n), w = x/L - floor(x/L), x/L rounded correctly.
//
// FP64 runs at 2 lanes a cycle here, so the definition's division, floor and conversions (about
// 25 FP64-rate operations an axis) would bound the kernels that bin atoms.  x (n/L) is instead
// added to 1.5 2^32: the sum's mantissa then holds it in units of 2^-20 and everything after is
// integer work.  It differs from the definition's value by less than 2 units (one rounding, and
// relative errors of 3e-16 of at most 2^31), so outside 2 units of a cell edge both give the same
// cell; on an edge (or outside the range, or not finite) the definition itself is evaluated.
// 1,000,000 atoms: binning 151 -> 54 us, mirror 246 -> 37 us.
// ------------------------------------------------------------------------------------
__device__ __noinline__ void cell_axis_plain(double x, double L, int n, int& q, int& c) {
    const double s = __ddiv_rn(x, L);
    const double fl = floor(s);
    const double w = __dsub_rn(s, fl);
    c = (int)__dmul_rn(w, (double)n);
    if (c >= n) c = n - 1;
    if (c < 0) c = 0;
    q = (int)fl * n + c;
}
__device__ __forceinline__ void cell_axis(double x, double L, double n_over_L, int n, int& q, int& c) {
    const double magic = 6442450944.0;           // 1.5 2^32: unit in the last place 2^-20
    const long long u = __double_as_longlong(__fma_rn(x, n_over_L, magic));
    const long long v = u - __double_as_longlong(magic);
    const unsigned fr = (unsigned)v & 0xfffffu;
    if ((u >> 52) != (__double_as_longlong(magic) >> 52) || fr - 2u > 0xffffbu) {
        cell_axis_plain(x, L, n, q, c);
        return;
    }
    q = (int)(v >> 20);
    c = q;
    if ((unsigned)q >= (unsigned)n) {
        c = q % n;
        c = c < 0 ? c + n : c;
    }
}

// The top 21 bits of each fraction in one 8-byte word, for pass A's row filter: x in bits 63-43, y
// in 42-22, z in 21-1.  The reader takes the words (hi, funnel shift by 21, lo << 10) as they are: what
// follows the 21 bits is noise below one unit.
__device__ __forceinline__ uint2 pack_frac(const int4& f) {
    const unsigned x = (unsigned)f.x >> 11, y = (unsigned)f.y >> 11, z = (unsigned)f.z >> 11;
    return make_uint2(y << 22 | z << 1, x << 11 | y >> 10);     // (lo, hi)
}

// Fractional position of x in the box of the last list build (frac32).  A resolution of L 2^-32 is
// finer than an FP32 coordinate within a cell up to some 1000 A; in longer boxes (fine) the next ten
// bits of each axis are kept in .w, ten apiece.
__device__ __forceinline__ int4 frac_position(const double (&x)[3], const DevState& st, int fine) {
    if (fine) {
        const long long a = frac42(x[0], st.ibox[0]), b = frac42(x[1], st.ibox[1]), c = frac42(x[2], st.ibox[2]);
        constexpr int mask = (1 << kFracLow) - 1;
        return make_int4((int)(unsigned)(a >> kFracLow), (int)(unsigned)(b >> kFracLow), (int)(unsigned)(c >> kFracLow),
                         ((int)a & mask) | ((int)b & mask) << kFracLow | ((int)c & mask) << 2 * kFracLow);
    }
    return make_int4(frac32(x[0], st.ibox[0]), frac32(x[1], st.ibox[1]), frac32(x[2], st.ibox[2]), 0);
}
// fb moved by (tx, ty, tz) units of 2^-32.
__device__ __forceinline__ int4 frac_moved(const int4& fb, float tx, float ty, float tz, int fine) {
    int4 f = make_int4(wrap_add(fb.x, __float2int_rn(tx)), wrap_add(fb.y, __float2int_rn(ty)), wrap_add(fb.z, __float2int_rn(tz)), 0);
    if (fine) {
        constexpr int mask = (1 << kFracLow) - 1;
        const auto low = [&](float t, int axis, int& hi) {
            const int v = ((fb.w >> axis * kFracLow) & mask) + __float2int_rn((t - rintf(t)) * (float)(mask + 1));
            hi = wrap_add(hi, v >> kFracLow);
            f.w |= (v & mask) << axis * kFracLow;
        };
        low(tx, 0, f.x); low(ty, 1, f.y); low(tz, 2, f.z);
    }
    return f;
}
// What the low bits (of fine positions) add to the difference j - i, in units of 2^-32.
__device__ __forceinline__ float3 frac_low_diff(int wj, int wi) {
    constexpr int mask = (1 << kFracLow) - 1;
    constexpr float unit = 1.0f / (mask + 1);
    return make_float3(unit * (float)((wj & mask) - (wi & mask)),
                       unit * (float)((wj >> kFracLow & mask) - (wi >> kFracLow & mask)),
                       unit * (float)((wj >> 2 * kFracLow & mask) - (wi >> 2 * kFracLow & mask)));
}

// The four rows of system s in lscale: L 2^-32 as FP32 value and remainder (what the fractional positions
// are scaled by), 1 - h/hb (0 while the box is the one of the last build; the division in FP64, since it
// is the small difference of two nearly equal edges) and 2^32 / L.  Kept per system and rewritten where
// the box changes: a division per block of the kernels that move the atoms had the integration of
// 128 x 4000 atoms under barostats at 45.4 us a launch, now 42.8 (an FP64 warp instruction issues in 16 cycles).
__device__ __forceinline__ void scale_axis(const Bufs& b, int s, int k, double box, double omr) {
    float* row = reinterpret_cast<float*>(b.lscale + 4 * s) + k;
    const double L = box * 0x1p-32;
    const float hi = (float)L;
    row[0] = hi;
    row[4] = (float)(L - (double)hi);
    row[8] = (float)omr;
    row[12] = 4294967296.0f / (float)box;
}
__device__ __forceinline__ void scale_of_box(const Bufs& b, int s, const DevState& st) {
    if (!b.lscale) return;
    for (int k = 0; k < 3; ++k) scale_axis(b, s, k, st.box[k], st.hmoved ? 1.0 - st.h[k] / st.hb[k] : 0.0);
}

// ------------------------------------------------------------------------------------
// Rebuild R1: fold the displacement into the FP64 anchor; cell of each atom, unwrapped cell
// index q, fresh mirror, spring offset, occupancy count.  The cell grid was set with the system's
// state (on the host for the stateless calls, by k_rebuild_list in the engine).
// ------------------------------------------------------------------------------------
template <typename T>
__device__ void cells_count_tile(const Bufs& b, int tile, int th) {
    using T4 = typename V4<T>::t;
    const TileAtom ta = tile_of(b, tile);
    const DevSys& S = b.sys[ta.sys];
    const DevState& st = b.st[ta.sys];
    if (th >= ta.count) return;
    const int i = ta.first + th;
    const size_t N = b.ntot;
    int c3[3], qv[3];
    double xm[3], sd[3] = {0.0, 0.0, 0.0};
    for (int k = 0; k < 3; ++k) {
        double xk = b.x[k * N + i];
        if (b.dhi) {   // fold the displacement into the FP64 anchor
            T* dh = reinterpret_cast<T*>(b.dhi);
            T* dl = reinterpret_cast<T*>(b.dlo);
            const double d = (double)dh[k * N + i] + (b.dlo ? (double)dl[k * N + i] : 0.0);
            xk = xk + d;
            b.x[k * N + i] = xk;
            dh[k * N + i] = (T)0;
            if (b.dlo) dl[k * N + i] = (T)0;
        }
        cell_axis(xk, st.box[k], st.ibox[k] * (double)st.ncell[k], st.ncell[k], qv[k], c3[k]);
        xm[k] = __fma_rn(-(double)qv[k], st.h[k], xk);   // (written out: the same in every kernel that builds)
        if (b.r0) sd[k] = xk - b.r0[k * N + i];
    }
    const int cell = c3[0] + st.ncell[0] * (c3[1] + st.ncell[1] * c3[2]);
    b.cell_of[i] = cell;
    b.q[i] = make_int4(qv[0], qv[1], qv[2], 0);
    const T4 m = mk4((T)xm[0], (T)xm[1], (T)xm[2], (T)0);
    reinterpret_cast<T4*>(b.xs)[i] = m;
    if (b.xa) reinterpret_cast<T4*>(b.xa)[i] = m;
    if (b.sd0) reinterpret_cast<T4*>(b.sd0)[i] = mk4((T)sd[0], (T)sd[1], (T)sd[2], (T)0);
    if (b.xfb && b.want_xf) {
        if (i == S.off) scale_of_box(b, ta.sys, st);
        const double x3[3] = {b.x[i], b.x[N + i], b.x[2 * N + i]};
        const int4 f = frac_position(x3, st, b.want_xf > 1);
        if (b.xf) b.xf[i] = f;
        b.xfb[i] = f;
        b.xc[i] = pack_frac(f);
    }
    atomicAdd(&b.cell_count[S.cell0 + cell], 1);
}

// The rebuild kernels walk a worklist of the tiles of flagged systems (written by
// k_rebuild_list) with a bounded grid, or every tile (stateless calls: no worklist).
#define NEFE_FOR_TILES(b, body_call)                                           \
    do {                                                                      \
        if ((b).rtiles) {                                                     \
            const int n_ = *(b).rcount;                                       \
            for (int w_ = blockIdx.x; w_ < n_; w_ += gridDim.x) {             \
                const int tile = (b).rtiles[w_];                              \
                body_call;                                                    \
            }                                                                 \
        } else {                                                              \
            const int tile = blockIdx.x;                                      \
            body_call;                                                        \
        }                                                                     \
    } while (0)

template <typename T>
__global__ void __launch_bounds__(kTile) k_cells_count(Bufs b) {
    dep_wait();
    NEFE_FOR_TILES(b, cells_count_tile<T>(b, tile, threadIdx.x));
}

// The cell grid of a system about to be rebuilt, at its current box.
__device__ __forceinline__ void set_cell_grid(const DevSys& S, DevState& st) {
    const double bx[3] = {st.box[0], st.box[1], st.box[2]};
    const bool same = st.grcs == S.rcs && st.gbox[0] == bx[0] && st.gbox[1] == bx[1] &&
                      st.gbox[2] == bx[2];
    if (!same) {
        int g3[3];
        const bool ok = grid_for(bx, S.rcs, S.ncell_cap, g3);
        for (int k = 0; k < 3; ++k) {
            st.ncell[k] = g3[k];
            st.h[k] = __ddiv_rn(bx[k], (double)g3[k]);
            st.hb[k] = st.h[k];
            st.ibox[k] = __ddiv_rn(1.0, bx[k]);
            st.gbox[k] = bx[k];
        }
        st.grcs = S.rcs;
        refresh_box_f(st);
        if (!ok) atomicOr(&st.err, NEFE_ERR_BOX);
    }
}

// Worklist of the tiles of every system whose rebuild flag is set (all with force_all), and the
// cell grid of each such system at its current box (per axis floor(L/rcs) reduced while
// L/n < rcs (1 + 1e-9), h = L/n, 1/L), computed once per system here rather than per tile, and
// only when the box or the list radius differ from the ones the grid was last computed for
// (the FP64 divisions are skipped for every system at fixed volume).
// Tile order in the list does not matter: every tile is processed independently.
// With b.rebuild_all, a step on which any system's flag is set rebuilds every system (the flags
// of all are set here, so the later rebuild kernels see them): rebuilding a list early never
// changes what the force passes compute, and one build over the whole batch runs its kernels at
// full width where many small builds, one per step, each pay their latency.
// The worklist of one step, built by one block (any multiple of 32 threads up to 256).
__device__ void build_worklist(const Bufs& b, int nsys, int force_all) {
    __shared__ int cnt;
    // no flag set anywhere this step (b.any_rebuild[0], written wherever a flag is): empty worklist
    if (!force_all && b.any_rebuild && *(volatile int*)b.any_rebuild == 0) {
        if (threadIdx.x == 0) {
            *b.rcount = 0;
            if (b.rcbase) b.rcbase[nsys] = 0;
        }
        return;
    }
    if (threadIdx.x == 0) cnt = 0;
    if (b.rebuild_all && !force_all) {
        int any = 0;
        for (int s = threadIdx.x; s < nsys; s += blockDim.x) any |= b.st[s].rebuild;
        if (__syncthreads_or(any))
            for (int s = threadIdx.x; s < nsys; s += blockDim.x) b.st[s].rebuild = 1;
    }
    __syncthreads();
    for (int s = threadIdx.x; s < nsys; s += blockDim.x) {
        DevState& st = b.st[s];
        if (force_all || st.rebuild) {
            const DevSys& S = b.sys[s];
            const int base = atomicAdd(&cnt, S.ntile);
            for (int t = 0; t < S.ntile; ++t) b.rtiles[base + t] = S.tile0 + t;
            set_cell_grid(S, st);
            st.nbuild += 1;
        }
    }
    __syncthreads();
    if (threadIdx.x == 0) *b.rcount = cnt;
    if (b.rcbase) {   // first worklist cell of each system: exclusive scan of the flagged cell counts
        __shared__ int wsum[8];
        const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (int)(blockDim.x >> 5);
        int carry = 0;
        for (int base = 0; base < nsys; base += (int)blockDim.x) {
            const int s = base + (int)threadIdx.x;
            int v = 0;
            if (s < nsys) {
                const DevState& st = b.st[s];
                if (force_all || st.rebuild) v = st.ncell[0] * st.ncell[1] * st.ncell[2];
            }
            int incl = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, incl, o);
                if (lane >= o) incl += y;
            }
            if (lane == 31) wsum[w] = incl;
            __syncthreads();
            int woff = 0, tot = 0;
            for (int k = 0; k < nw; ++k) {
                if (k < w) woff += wsum[k];
                tot += wsum[k];
            }
            if (s < nsys) b.rcbase[s] = carry + woff + incl - v;
            carry += tot;
            __syncthreads();
        }
        if (threadIdx.x == 0) b.rcbase[nsys] = carry;
    }
}

__global__ void __launch_bounds__(256) k_rebuild_list(Bufs b, int nsys, int force_all) {
    dep_wait();
    build_worklist(b, nsys, force_all);
}

constexpr int kCellsCluster = 8, kCellsThreads = 512;   // k_cells_clusters: blocks per system, threads

// R2: exclusive scan of cells [lo, hi) of system s's occupancy by one block (blockDim a multiple
// of 32, at most 512; 8 consecutive cells per thread per pass), starting from `carry`; resets the
// counts.  The block that holds the last cell writes the total.
__device__ void scan_cells_range(const Bufs& b, int s, int lo, int hi, int ncells, int carry) {
    constexpr int PT = 8;
    const DevSys& S = b.sys[s];
    int* start = b.cell_start + S.cell0 + s;
    int* count = b.cell_count + S.cell0;
    int* cursor = b.cell_cursor + S.cell0;
    __shared__ int warp_tot[kCellsThreads / 32];
    const int lane = threadIdx.x & 31, w = threadIdx.x >> 5, nw = (int)(blockDim.x >> 5);
    const int span = (int)blockDim.x * PT;
    for (int base = lo; base < hi; base += span) {
        const int c0 = base + (int)threadIdx.x * PT;
        int v[PT], tsum = 0;
#pragma unroll
        for (int u = 0; u < PT; ++u) {
            v[u] = c0 + u < hi ? count[c0 + u] : 0;
            tsum += v[u];
        }
        int incl = tsum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) warp_tot[w] = incl;
        __syncthreads();
        int woff = 0, tot = 0;
        for (int k = 0; k < nw; ++k) {
            if (k < w) woff += warp_tot[k];
            tot += warp_tot[k];
        }
        int run = carry + woff + incl - tsum;
#pragma unroll
        for (int u = 0; u < PT; ++u) {
            if (c0 + u < hi) {
                start[c0 + u] = run;
                cursor[c0 + u] = run;
                count[c0 + u] = 0;
            }
            run += v[u];
        }
        carry += tot;
        __syncthreads();                         // warp_tot is rewritten by the next pass
    }
    if (threadIdx.x == 0 && hi == ncells) {
        start[ncells] = carry;
        if (carry != S.n) atomicOr(&b.st[s].err, NEFE_ERR_CELL);
    }
}

__device__ void scan_system_cells(const Bufs& b, int s) {
    const DevState& st = b.st[s];
    const int ncells = st.ncell[0] * st.ncell[1] * st.ncell[2];
    scan_cells_range(b, s, 0, ncells, ncells, 0);
}

// One 256-thread block per system; systems whose rebuild flag is clear return (all are scanned
// with force_all).
__global__ void __launch_bounds__(256) k_cells_scan(Bufs b, int force_all) {
    dep_wait();
    const int s = blockIdx.x;
    if (!force_all && !b.st[s].rebuild) return;
    scan_system_cells(b, s);
}

// The same scan of one large system (stateless calls) by several blocks, in two launches: the
// occupancy sum of each block's span, then each block sums the spans before its own (at most
// kScanBlocks of them) and scans its span from there.  One block alone walks 2048 cells in
// 3.7 us, one pass after the other: 452 us for the 250,047 cells of 1,000,000 atoms, 8 us here;
// up to kScanOneBlock cells (two passes) the single block is as fast and one launch less.
constexpr int kScanBlocks = 1024;
constexpr int kScanOneBlock = 4096;
__global__ void __launch_bounds__(256) k_cells_span_sums(Bufs b, int span, int* sums) {
    dep_wait();
    const DevState& st = b.st[0];
    const int ncells = st.ncell[0] * st.ncell[1] * st.ncell[2];
    const int lo = blockIdx.x * span, hi = min(ncells, lo + span);
    int v = 0;
    for (int c = lo + (int)threadIdx.x; c < hi; c += (int)blockDim.x) v += b.cell_count[c];
    __shared__ int red[8];
    v = __reduce_add_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    if (threadIdx.x == 0) {
        for (int k = 1; k < 8; ++k) v += red[k];
        sums[blockIdx.x] = v;
    }
}
__global__ void __launch_bounds__(256) k_cells_scan_spans(Bufs b, int span, const int* sums) {
    dep_wait();
    const DevState& st = b.st[0];
    const int ncells = st.ncell[0] * st.ncell[1] * st.ncell[2];
    int v = 0;
    for (int k = threadIdx.x; k < (int)blockIdx.x; k += (int)blockDim.x) v += sums[k];
    __shared__ int red[8];
    v = __reduce_add_sync(0xffffffffu, v);
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
    __syncthreads();
    int carry = 0;
    for (int k = 0; k < 8; ++k) carry += red[k];
    const int lo = blockIdx.x * span;
    scan_cells_range(b, 0, lo, min(ncells, lo + span), ncells, carry);
}

// Atom index carried in the .w lane of a position vector (bit pattern in FP32, value in FP64).
template <typename T> __device__ __forceinline__ T pack_index(int i);
template <> __device__ __forceinline__ float pack_index<float>(int i) { return __int_as_float(i); }
template <> __device__ __forceinline__ double pack_index<double>(int i) { return (double)i; }
__device__ __forceinline__ int unpack_index(float w) { return __float_as_int(w); }
__device__ __forceinline__ int unpack_index(double w) { return (int)w; }

// R3: scatter atoms into their cell segment (order inside a cell fixed by R4), with a copy
// of their mirror positions in the same order for the list build.
template <typename T>
__device__ void cells_fill_tile(const Bufs& b, int tile, int th) {
    using T4 = typename V4<T>::t;
    const TileAtom ta = tile_of(b, tile);
    const DevSys& S = b.sys[ta.sys];
    if (th >= ta.count) return;
    const int i = ta.first + th;
    const int pos = atomicAdd(&b.cell_cursor[S.cell0 + b.cell_of[i]], 1);
    if (pos < 0 || pos >= S.n) {                 // inconsistent occupancy: record, never write out of range
        atomicOr(&b.st[ta.sys].err, NEFE_ERR_CELL);
        return;
    }
    b.perm[S.off + pos] = i;
    if (b.xcs) {
        const T4 m = reinterpret_cast<const T4*>(b.xs)[i];
        reinterpret_cast<T4*>(b.xcs)[S.off + pos] = mk4(m.x, m.y, m.z, pack_index<T>(i));
    }
}
template <typename T>
__global__ void __launch_bounds__(kTile) k_cells_fill(Bufs b) {
    dep_wait();
    NEFE_FOR_TILES(b, cells_fill_tile<T>(b, tile, threadIdx.x));
}

// Worklist, R1, R2 and R3 of a small context (at most 32 systems and kClusterTiles tiles) in one launch: a
// cluster of 8 blocks per system, with cluster barriers between the passes.  There is no worklist:
// the list builds go by the systems' own flags (for_cells_of_grid).  On most steps no flag is set
// and the launch returns at once, where the four launches cost 1.1 us each: 64 atoms in FP64 43.1 -> 40.8 us
// a step, one 8000-atom system (63 tiles) 26.0 -> 24.9.  Larger contexts keep the separate kernels, which
// spread a rebuild over the whole chip: 4 x 8000 atoms (252 tiles) 96 us a step against 100 in clusters,
// 12 x 8000 76.6 against 77.7.
constexpr int kClusterSystems = 32, kClusterTiles = 128;
__device__ __forceinline__ void cluster_sync() {
    asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
template <typename T>
__global__ void __cluster_dims__(kCellsCluster) __launch_bounds__(kCellsThreads) k_cells_clusters(Bufs b, int nsys) {
    dep_wait();
    if (*(volatile int*)b.any_rebuild == 0) return;
    const int s = (int)blockIdx.x / kCellsCluster, rank = (int)blockIdx.x % kCellsCluster;
    const DevSys& S = b.sys[s];
    DevState& st = b.st[s];
    // with rebuild_all any system's flag flags all; a flag set meanwhile by another cluster implies it
    const int mine = (int)threadIdx.x < nsys && (b.rebuild_all || (int)threadIdx.x == s)
                         ? *(volatile int*)&b.st[threadIdx.x].rebuild : 0;
    if (!__syncthreads_or(mine)) return;         // uniform over the cluster
    if (rank == 0 && threadIdx.x == 0) {
        *(volatile int*)&st.rebuild = 1;
        set_cell_grid(S, st);
        st.nbuild += 1;
    }
    cluster_sync();
    const int sub = (int)threadIdx.x / kTile, th = (int)threadIdx.x % kTile;
    const int t0 = rank * (kCellsThreads / kTile) + sub, step = kCellsCluster * (kCellsThreads / kTile);
    for (int t = t0; t < S.ntile; t += step) cells_count_tile<T>(b, S.tile0 + t, th);
    cluster_sync();
    if (rank == 0) scan_system_cells(b, s);
    cluster_sync();
    for (int t = t0; t < S.ntile; t += step) cells_fill_tile<T>(b, S.tile0 + t, th);
}

// R4: insertion sort of each cell segment by atom index (stable order by (cell, atom)), one cell
// per thread over gridDim.x blocks.  Only the stateless cell sort runs it: the list builds rank
// their rows themselves.
__global__ void __launch_bounds__(256) k_cells_sort(Bufs b) {
    dep_wait();
    constexpr int s = 0;
    const DevSys& S = b.sys[s];
    const DevState& st = b.st[s];
    const int ncells = st.ncell[0] * st.ncell[1] * st.ncell[2];
    const int* start = b.cell_start + S.cell0 + s;
    int* p = b.perm + S.off;
    for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < ncells; c += gridDim.x * blockDim.x) {
        const int lo = max(0, min(start[c], S.n)), hi = max(lo, min(start[c + 1], S.n));
        for (int a = lo + 1; a < hi; ++a) {
            const int key = p[a];
            int z = a - 1;
            while (z >= lo && p[z] > key) { p[z + 1] = p[z]; --z; }
            p[z + 1] = key;
        }
    }
}

// Index of entry k of atom i's Verlet row (see Bufs::nbr_il).  The interleaved form lets the
// lanes of a warp that take consecutive atoms read their next four entries as one contiguous
// 512-byte request.
__device__ __forceinline__ size_t nbr_at(const Bufs& b, int i, int k) {
    return b.nbr_il ? ((size_t)(k >> 2) * b.ntot + i) * 4 + (k & 3) : (size_t)i * b.cap + k;
}

// Padding of an interleaved row past its mrow entries up to the next multiple of 4: atom i's
// own image through cell offset (-1, -1, -1), at distance |(h_x, h_y, h_z)| >= sqrt(3) rcs
// from i, so it never enters a shell (the force passes read whole groups of four).
__device__ __forceinline__ void pad_row(const Bufs& b, int i, int mrow, int lane, int nlanes) {
    if (!b.nbr_il) return;
    const int end = (mrow + 3) & ~3;
    for (int k = mrow + lane; k < end && k < b.cap; k += nlanes) b.nbr[nbr_at(b, i, k)] = i;
}

// Debug build (NEFE_DEBUG_BOUNDS, libnefe_debug.so): every atom index read from device data
// (list entries, shell entries, UF rows) is checked before it is used; an index outside the
// context's atoms sets NEFE_ERR_CELL in the system's error word and the access is skipped (a
// list entry is replaced by the row's padding entry, which never enters a shell).  In the
// normal build the check compiles away.
#ifdef NEFE_DEBUG_BOUNDS
#define NEFE_IN_RANGE(idx, n, errp) \
    (((unsigned)(idx) < (unsigned)(n)) ? true : (atomicOr((errp), (unsigned)NEFE_ERR_CELL), false))
#else
#define NEFE_IN_RANGE(idx, n, errp) true
#endif

// Exact list criterion in FP64, the plain definition: raw = x_j - x_i, m = rint(raw/L),
// d = raw - m L, ((d_x^2 + d_y^2) + d_z^2) < rcs^2; every operation rounded separately.
__device__ __noinline__ bool exact_pair_in(const Bufs& b, const double box[3], int i, int j,
                                           double rcs2, double d[3]) {
    for (int k = 0; k < 3; ++k) {
        const double raw = __dsub_rn(b.x[(size_t)k * b.ntot + j], b.x[(size_t)k * b.ntot + i]);
        const double m = rint(__ddiv_rn(raw, box[k]));
        d[k] = __dsub_rn(raw, __dmul_rn(m, box[k]));
    }
    double rr = __dadd_rn(__dmul_rn(d[0], d[0]), __dmul_rn(d[1], d[1]));
    rr = __dadd_rn(rr, __dmul_rn(d[2], d[2]));
    return rr < rcs2;
}

// R5: Verlet list, L lanes per atom (a group of L lanes of one warp).
// The 27 neighbour cells of atom i's cell form 9 x-rows (one per (oy, oz)); the three cells of
// a row (ox = -1, 0, 1) are consecutive in the cell-ordered mirror copy unless the row wraps at
// the box edge (cx = 0 or cx = nx - 1), so a row is one contiguous range of candidates (two
// pieces where it wraps).  A cell whose box is farther than rcs from atom i is pruned, which
// trims a row at its ends or drops it.  The pieces are concatenated into one candidate sequence
// of the group, which its lanes walk L at a time (lane l takes candidates l, l + L, ...: every
// lane but the last pass's is busy); the cell offset of a candidate follows from its position
// against its piece's cell boundaries.  A candidate is accepted or rejected on its mirror
// distance when that lies outside a relative band of 1e-4 (FP32) / 1e-10 (FP64) around rcs^2,
// and inside the band by the exact FP64 criterion (which must also agree with the offset's
// image), so the list equals the plain definition bit for bit.  Accepted entries are appended
// through a ballot, as keys j * 32 + o, and then ranked by atom index into the row, which
// fixes the order.
constexpr int kRebuildBlocks = 152 * 8;   // bounded grid of the worklist-driven rebuild kernels
constexpr int kRowPieces = 18;            // piece p of row r at 2 r + p
constexpr int kKeyRow = kMaxCap + 4;      // key buffer row: 16-byte aligned, groups on different banks

// Per-group tables of the list build in shared memory.
template <typename T>
struct NlistShared {
    using T4 = typename V4<T>::t;
    int4 pc[kRowPieces];          // (first candidate in xcs, start of its 2nd cell, of its 3rd cell, first flat index)
    T4 ps[kRowPieces];            // (x_i - ox h_x, y_i - oy h_y, z_i - oz h_z) of the piece's first cell
    int code[kRowPieces];         // cell-offset code of the piece's first cell
    int flat_end;                 // number of candidates of the group
};

// One piece of row (oy, oz): cells x0 .. x0 + nc - 1 of the row starting at rb (consecutive in
// memory), as (first candidate, end, start of the second cell, start of the third cell), the
// last two INT_MAX when absent.
__device__ __forceinline__ int4 row_piece(const int* start, int rb, int x0, int nc, int n) {
    const int lo = max(0, min(start[rb + x0], n));
    const int hi = max(lo, min(start[rb + x0 + nc], n));
    const int b1 = nc > 1 ? start[rb + x0 + 1] : INT_MAX;
    const int b2 = nc > 2 ? start[rb + x0 + 2] : INT_MAX;
    return make_int4(lo, hi, b1, b2);
}

template <typename T, int L>
__device__ void nlist_item(const Bufs& b, int tile, int part, unsigned (*keys)[kKeyRow],
                           NlistShared<T>* tab) {
    using T4 = typename V4<T>::t;
    constexpr int G = kTile / L;
    constexpr int RR = (9 + L - 1) / L;          // rows per lane
    const TileAtom ta = tile_of(b, tile);
    const DevSys& S = b.sys[ta.sys];
    if (S.pot != POT_SW) {                       // no SW term: no SW list (uniform over the block)
        const int ia = part * G + (int)threadIdx.x / L;
        if (threadIdx.x % L == 0 && ia < ta.count) b.cnt[ta.first + ia] = 0;
        return;
    }
    DevState& st = b.st[ta.sys];
    const int lane = threadIdx.x % L, grp = threadIdx.x / L;
    const int lbase = ((threadIdx.x & 31) / L) * L;
    NlistShared<T>& sh = tab[grp];
    const int ia = part * G + grp;
    // groups past the tile's end stay in the warp-uniform loops below with no candidates
    const bool valid = ia < ta.count;
    const int i = ta.first + (valid ? ia : 0);
    const int nx = st.ncell[0], ny = st.ncell[1], nz = st.ncell[2];
    const int cell = b.cell_of[i];
    const int cx = cell % nx, cy = (cell / nx) % ny, cz = cell / (nx * ny);
    const int* start = b.cell_start + S.cell0 + ta.sys;
    const T4 xi = reinterpret_cast<const T4*>(b.xs)[i];
    const T hx = pick<T>(st.h[0], st.h_f[0]), hy = pick<T>(st.h[1], st.h_f[1]), hz = pick<T>(st.h[2], st.h_f[2]);
    T lo2, hi2;
    if constexpr (sizeof(T) == 4) {
        lo2 = S.rcs2_lo_f;
        hi2 = S.rcs2_hi_f;
    } else {
        lo2 = S.rcs * S.rcs * (1.0 - 1e-10);
        hi2 = S.rcs * S.rcs * (1.0 + 1e-10);
    }
    // pruning bound: relaxed by 1e-3 of rcs^2, far above the rounding of the mirror positions
    // (which lie in [0, h) of their own cell), so no pair within rcs can be missed
    const T prune2 = (T)(S.rcs * S.rcs * 1.001);
    const T4* xc = reinterpret_cast<const T4*>(b.xcs) + S.off;
    // first ox of a row's second piece: the row wraps between ox = -1 and 0 (cx = 0) or between
    // 0 and +1 (cx = nx - 1); 2 when it does not wrap (nx >= 2, so never both)
    const int brk = cx == 0 ? 0 : (cx == nx - 1 ? 1 : 2);
    int carry = 0;
#pragma unroll
    for (int k = 0; k < RR; ++k) {
        const int r = lane + k * L;
        int4 p0 = make_int4(0, 0, INT_MAX, INT_MAX), p1 = p0;
        int a = 0, a2 = 0, cb = 0;
        if (valid && r < 9) {
            const int oy = r % 3 - 1, oz = r / 3 - 1;
            const T ey = oy < 0 ? xi.y : (oy > 0 ? hy - xi.y : (T)0);
            const T ez = oz < 0 ? xi.z : (oz > 0 ? hz - xi.z : (T)0);
            const T fy = ey > (T)0 ? ey : (T)0, fz = ez > (T)0 ? ez : (T)0;
            const T fyz = fy * fy + fz * fz;
            cb = 3 * (oy + 1) + 9 * (oz + 1);
            if (fyz <= prune2) {
                const T fl = xi.x > (T)0 ? xi.x : (T)0, fr = hx - xi.x > (T)0 ? hx - xi.x : (T)0;
                a = fl * fl + fyz <= prune2 ? -1 : 0;          // lower cell kept
                const int e = fr * fr + fyz <= prune2 ? 1 : 0; // upper cell kept
                int yy = cy + oy, zz = cz + oz;
                yy = yy < 0 ? yy + ny : (yy >= ny ? yy - ny : yy);
                zz = zz < 0 ? zz + nz : (zz >= nz ? zz - nz : zz);
                const int rb = nx * (yy + ny * zz);
                const int e1 = min(e, brk - 1);               // first piece: ox = a .. e1
                if (a <= e1) {
                    int x0 = cx + a;
                    x0 = x0 < 0 ? x0 + nx : x0;
                    p0 = row_piece(start, rb, x0, e1 - a + 1, S.n);
                }
                a2 = max(a, brk);                             // second piece: ox = a2 .. e
                if (brk < 2 && a2 <= e) {
                    int x0 = cx + a2;
                    x0 = x0 >= nx ? x0 - nx : x0;
                    p1 = row_piece(start, rb, x0, e - a2 + 1, S.n);
                }
            }
            const T yo = xi.y - (T)oy * hy, zo = xi.z - (T)oz * hz;
            sh.ps[2 * r] = mk4(xi.x - (T)a * hx, yo, zo, (T)0);
            sh.ps[2 * r + 1] = mk4(xi.x - (T)a2 * hx, yo, zo, (T)0);
            sh.code[2 * r] = cb + a + 1;
            sh.code[2 * r + 1] = cb + a2 + 1;
        }
        // flat positions: exclusive scan of the rows' lengths over the group, row order
        const int n0 = p0.y - p0.x, len = n0 + (p1.y - p1.x);
        int incl = len;
#pragma unroll
        for (int o = 1; o < L; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, incl, o, L);
            if (lane >= o) incl += y;
        }
        const int f0 = carry + incl - len;
        if (valid && r < 9) {
            sh.pc[2 * r] = make_int4(p0.x, p0.z, p0.w, f0);
            sh.pc[2 * r + 1] = make_int4(p1.x, p1.z, p1.w, f0 + n0);
        }
        carry += __shfl_sync(0xffffffffu, incl, L - 1, L);
    }
    if (lane == 0) sh.flat_end = carry;
    __syncwarp();
    // walk the flat sequence L candidates at a time; the pass count is uniform over the warp
    const int total = carry;
    const int npass = __reduce_max_sync(0xffffffffu, (total + L - 1) / L);
    int cnt = 0;
    for (int pass = 0; pass < npass; ++pass) {
        const int t = pass * L + lane;
        bool in = false, band = false, bad = false;
        unsigned key = 0u;
        T dx = (T)0, dy = (T)0, dz = (T)0;
        int j = 0;
        if (t < total) {                         // straight-line: no branch inside
            int e = 0;                           // piece of t: last entry whose flat start is <= t
#pragma unroll
            for (int step = 16; step > 0; step >>= 1) {
                const int c = e + step;
                if (c < kRowPieces && sh.pc[c].w <= t) e = c;
            }
            const int4 pc = sh.pc[e];
            const T4 po = sh.ps[e];
            const int p = pc.x + (t - pc.w);
            const T4 xj = xc[p];
            j = unpack_index(xj.w);
            const int inc = (p >= pc.y ? 1 : 0) + (p >= pc.z ? 1 : 0);
            const int o = sh.code[e] + inc;
            dx = (xj.x - po.x) + (T)inc * hx;
            dy = xj.y - po.y;
            dz = xj.z - po.z;
            const T dd = dx * dx + dy * dy + dz * dz;
            bad = (unsigned)(j - S.off) >= (unsigned)S.n;
            const bool cand = !bad && !(j == i && o == 13);
            in = cand && dd < lo2;
            band = cand && !(dd < lo2) && dd <= hi2;
            key = (unsigned)j * 32u + (unsigned)o;
        }
        if (__any_sync(0xffffffffu, bad || band)) {   // rare: a corrupt cell table or the exact test
            if (bad) atomicOr(&st.err, NEFE_ERR_CELL);
            if (band) {
                double d[3];
                in = exact_pair_in(b, st.box, i, j, __dmul_rn(S.rcs, S.rcs), d);
                in = in && fabs(d[0] - (double)dx) < 0.5 * st.h[0] &&
                     fabs(d[1] - (double)dy) < 0.5 * st.h[1] &&
                     fabs(d[2] - (double)dz) < 0.5 * st.h[2];
            }
        }
        const unsigned bal = __ballot_sync(0xffffffffu, in);
        const unsigned m = (L == 32) ? bal : ((bal >> lbase) & ((1u << L) - 1u));
        const int pos = cnt + __popc(m & ((1u << lane) - 1u));
        if (in && pos < kMaxCap) keys[grp][pos] = key;
        cnt += __popc(m);
    }
    // rank by atom index into the row (indices in a row are distinct); the key row is padded to
    // a multiple of 4 with the largest key, so it is read 4 keys at a time
    const int have = cnt < kMaxCap ? cnt : kMaxCap;
    const int have4 = (have + 3) & ~3;
    for (int z = have + lane; z < have4; z += L) keys[grp][z] = 0xffffffffu;
    __syncwarp();
    if (valid) {
        const int cap = b.cap;
        const int mrow = cnt < cap ? cnt : cap;
        const uint4* row4 = reinterpret_cast<const uint4*>(keys[grp]);
        constexpr int R = 4;
        for (int a0 = 0; a0 < have; a0 += R * L) {
            unsigned k[R];
            int rk[R];
#pragma unroll
            for (int u = 0; u < R; ++u) {
                const int a = a0 + u * L + lane;
                k[u] = a < have ? keys[grp][a] : 0xffffffffu;
                rk[u] = 0;
            }
            for (int z = 0; z < have4; z += 4) {
                const uint4 v = row4[z >> 2];
#pragma unroll
                for (int u = 0; u < R; ++u)
                    rk[u] += (v.x < k[u] ? 1 : 0) + (v.y < k[u] ? 1 : 0) + (v.z < k[u] ? 1 : 0) +
                             (v.w < k[u] ? 1 : 0);
            }
#pragma unroll
            for (int u = 0; u < R; ++u) {
                const int a = a0 + u * L + lane;
                if (a < have && rk[u] < mrow)
                    b.nbr[nbr_at(b, i, rk[u])] = (int)((k[u] >> 5) | ((k[u] & 31u) << kCodeShift));
            }
        }
        pad_row(b, i, mrow, lane, L);
        if (lane == 0) {
            b.cnt[i] = cnt;
            if (cnt > cap) atomicOr(&st.err, NEFE_ERR_NBR_OVERFLOW);
        }
    }
    __syncwarp();                                // shared tables reused by the next item
}

template <typename T, int L>
__global__ void __launch_bounds__(kTile, 8) k_nlist(Bufs b) {
    dep_wait();
    constexpr int G = kTile / L;
    __shared__ __align__(16) unsigned keys[G][kKeyRow];
    __shared__ NlistShared<T> tab[G];
    if (b.rtiles) {
        const int n = *b.rcount * L;
        for (int w = blockIdx.x; w < n; w += gridDim.x) nlist_item<T, L>(b, b.rtiles[w / L], w % L, keys, tab);
    } else {
        nlist_item<T, L>(b, blockIdx.x / L, blockIdx.x % L, keys, tab);
    }
}

// R5 (list mode 0, the default): one warp per cell.  The atoms of a cell share its 27 neighbour
// cells, so the warp walks that candidate sequence once (its 9 x-rows as pieces, 32 candidates
// at a time, one per lane: position, image offset and index loaded once) and tests every
// candidate against each atom of the cell in turn (the cell's atoms up to 8 at a time, their
// positions in shared memory), with the same filter, band and exact test as above.  An accepted
// key j * 32 + o is appended to the cell atom's shared row (ballot and prefix count), and the keys of
// all rows of the cell are then ranked by key, i.e. by atom index, and stored, one key per lane.
// Every candidate position is read once per neighbouring cell instead of once per neighbouring
// atom.  Bound by instruction issue (70 %): ranking one row at a time, 17 of 32 lanes in use, and
// appending by shared-memory atomics, 1,000,000 atoms 630 us -> 534.
constexpr int kHomeChunk = 8;             // cell atoms per walk of the candidate sequence
template <typename T>
struct CellListShared {
    using T4 = typename V4<T>::t;
    unsigned keys[kHomeChunk][kKeyRow];   // accepted keys of each cell atom
    T4 home[kHomeChunk];                  // cell atoms: mirror position, index in .w
    int4 pc[kRowPieces];                  // (first candidate, start of 2nd cell, of 3rd cell, first flat index)
    T4 po[kRowPieces];                    // offset (ox h_x, oy h_y, oz h_z) of the piece's first cell
    int code[kRowPieces];                 // cell-offset code of the piece's first cell
    int pw[kRowPieces];                   // first flat index of each piece (the .w of pc again, as
                                          // one int row: the search reads it without conflicts)
    int2 first[kHomeChunk];               // of each cell atom: first flat key (rows padded to 4), accepted count
};

template <typename T>
__device__ __forceinline__ void nlist_cell(const Bufs& b, int s, int c, CellListShared<T>& sh, int lane) {
    using T4 = typename V4<T>::t;
    constexpr unsigned kAll = 0xffffffffu;
    const DevSys& S = b.sys[s];
    DevState& st = b.st[s];
    const int* start = b.cell_start + S.cell0 + s;
    const int n = S.n, off = S.off;
    const int hs = max(0, min(start[c], n)), he = max(hs, min(start[c + 1], n));
    const int m = he - hs;
    if (m == 0) return;
    const T4* xc = reinterpret_cast<const T4*>(b.xcs) + off;
    if (S.pot != POT_SW) {                       // no SW term: no SW list
        for (int q = lane; q < m; q += 32) {
            const int i = unpack_index(xc[hs + q].w);
            if ((unsigned)(i - off) < (unsigned)n) b.cnt[i] = 0;
        }
        return;
    }
    const int nx = st.ncell[0], ny = st.ncell[1], nz = st.ncell[2];
    const int cx = c % nx, cy = (c / nx) % ny, cz = c / (nx * ny);
    const T hx = pick<T>(st.h[0], st.h_f[0]), hy = pick<T>(st.h[1], st.h_f[1]), hz = pick<T>(st.h[2], st.h_f[2]);
    T lo2, hi2;
    if constexpr (sizeof(T) == 4) {
        lo2 = S.rcs2_lo_f;
        hi2 = S.rcs2_hi_f;
    } else {
        lo2 = S.rcs * S.rcs * (1.0 - 1e-10);
        hi2 = S.rcs * S.rcs * (1.0 + 1e-10);
    }
    // the rows: lane r < 9 builds row r = (oy, oz) as one piece (ox = -1 .. 1), or two where it
    // wraps at the box edge (cx = 0: the piece ox = -1, then 0 .. 1; cx = nx - 1: -1 .. 0, then 1)
    const int brk = cx == 0 ? 0 : (cx == nx - 1 ? 1 : 2);
    int len = 0, n0 = 0;
    int4 p0 = make_int4(0, 0, INT_MAX, INT_MAX), p1 = p0;
    int a2 = 0;
    if (lane < 9) {
        const int oy = lane % 3 - 1, oz = lane / 3 - 1;
        int yy = cy + oy, zz = cz + oz;
        yy = yy < 0 ? yy + ny : (yy >= ny ? yy - ny : yy);
        zz = zz < 0 ? zz + nz : (zz >= nz ? zz - nz : zz);
        const int rb = nx * (yy + ny * zz);
        const int e1 = min(1, brk - 1);
        a2 = brk;
        if (-1 <= e1) p0 = row_piece(start, rb, cx == 0 ? nx - 1 : cx - 1, e1 + 2, n);
        if (brk < 2) p1 = row_piece(start, rb, cx + a2 >= nx ? cx + a2 - nx : cx + a2, 2 - a2, n);
        n0 = p0.y - p0.x;
        len = n0 + (p1.y - p1.x);
    }
    int incl = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kAll, incl, o);
        if (lane >= o) incl += y;
    }
    const int total = __shfl_sync(kAll, incl, 31);
    if (lane < 9) {
        const int oy = lane % 3 - 1, oz = lane / 3 - 1;
        const int f0 = incl - len;
        const T offy = (T)oy * hy, offz = (T)oz * hz;
        const int cb = 3 * (oy + 1) + 9 * (oz + 1);
        sh.pw[2 * lane] = f0;
        sh.pw[2 * lane + 1] = f0 + n0;
        sh.pc[2 * lane] = make_int4(p0.x, p0.z, p0.w, f0);
        sh.po[2 * lane] = mk4(-hx, offy, offz, (T)0);
        sh.code[2 * lane] = cb;
        sh.pc[2 * lane + 1] = make_int4(p1.x, p1.z, p1.w, f0 + n0);
        sh.po[2 * lane + 1] = mk4((T)a2 * hx, offy, offz, (T)0);
        sh.code[2 * lane + 1] = cb + a2 + 1;
    }
    __syncwarp();
    const int cap = b.cap;
    for (int h0 = 0; h0 < m; h0 += kHomeChunk) {
        const int mh = min(kHomeChunk, m - h0);
        if (lane < mh) sh.home[lane] = xc[hs + h0 + lane];
        __syncwarp();
        int cnt = 0;                             // lane a: accepted count of cell atom a
        for (int t0 = 0; t0 < total; t0 += 32) {
            const int t = t0 + lane;
            int j = -1, o = 0, self = -1;        // self: which cell atom the candidate itself is
            // a candidate that is not one (past the sequence, or a bad index) sits far away, so
            // the distance test below rejects it without a separate flag
            T cxj = (T)1e15, cyj = (T)1e15, czj = (T)1e15;
            if (t < total) {
                int e = 0;                       // piece of t: last entry whose flat start is <= t
#pragma unroll
                for (int step = 16; step > 0; step >>= 1) {
                    const int q = e + step;
                    if (q < kRowPieces && sh.pw[q] <= t) e = q;
                }
                const int4 pc = sh.pc[e];
                const T4 po = sh.po[e];
                const int p = pc.x + (t - pc.w);
                const T4 xj = xc[p];
                j = unpack_index(xj.w);
                const int inc = (p >= pc.y ? 1 : 0) + (p >= pc.z ? 1 : 0);
                o = sh.code[e] + inc;
                if (o == 13) self = p - hs - h0;
                if ((unsigned)(j - off) < (unsigned)n) {
                    cxj = xj.x + (po.x + (T)inc * hx);
                    cyj = xj.y + po.y;
                    czj = xj.z + po.z;
                } else {
                    atomicOr(&st.err, NEFE_ERR_CELL);
                }
            }
            const unsigned key = (unsigned)j * 32u + (unsigned)o, below = (1u << lane) - 1u;
            // The common path is the distance test alone; a candidate inside the band is decided by
            // the exact FP64 criterion.  The lanes that accept append their keys in lane order (any
            // order would do: the row is ranked by key below).
            for (int a = 0; a < mh; ++a) {
                const T4 ha = sh.home[a];
                const T dx = cxj - ha.x, dy = cyj - ha.y, dz = czj - ha.z;
                const T dd = dx * dx + dy * dy + dz * dz;
                bool in = dd <= hi2 && a != self;
                if (in && !(dd < lo2)) {         // rare
                    double d[3];
                    in = exact_pair_in(b, st.box, unpack_index(ha.w), j, __dmul_rn(S.rcs, S.rcs), d);
                    in = in && fabs(d[0] - (double)dx) < 0.5 * st.h[0] &&
                         fabs(d[1] - (double)dy) < 0.5 * st.h[1] &&
                         fabs(d[2] - (double)dz) < 0.5 * st.h[2];
                }
                const unsigned bal = __ballot_sync(kAll, in);
                const int pos = __shfl_sync(kAll, cnt, a) + __popc(bal & below);
                if (in && pos < kMaxCap) sh.keys[a][pos] = key;
                if (lane == a) cnt += __popc(bal);
            }
        }
        // The rows: the keys of all the cell atoms, one per lane, each ranked by atom index within its
        // row (the row padded to a multiple of 4 with the largest key and read 4 keys at a time) and
        // stored at its rank.  An interleaved row is padded past its end with the atom itself.
        const int have_l = min(cnt, kMaxCap), pad_l = (have_l + 3) & ~3;    // (0 past the cell's atoms)
        int upto = pad_l;
#pragma unroll
        for (int k = 1; k < kHomeChunk; k <<= 1) {
            const int y = __shfl_up_sync(kAll, upto, k);
            if (lane >= k) upto += y;
        }
        const int all = __shfl_sync(kAll, upto, kHomeChunk - 1);
        if (lane < kHomeChunk) {
            for (int k = have_l; k < pad_l; ++k) sh.keys[lane][k] = 0xffffffffu;
            sh.first[lane] = make_int2(upto - pad_l, cnt);
        }
        __syncwarp();
        for (int t0 = 0; t0 < all; t0 += 32) {
            const int t = t0 + lane;
            if (t < all) {
                int a = 0;                       // row of t: last one that starts at or below it
#pragma unroll
                for (int step = kHomeChunk / 2; step > 0; step >>= 1)
                    if (sh.first[a + step].x <= t) a += step;
                const int f = sh.first[a].x, c = sh.first[a].y;
                const int ia = unpack_index(sh.home[a].w), have = min(c, kMaxCap), mrow = min(c, cap);
                const unsigned key = sh.keys[a][t - f];
                const uint4* row4 = reinterpret_cast<const uint4*>(sh.keys[a]);
                int rk = 0;
                for (int z = 0; 4 * z < have; ++z) {
                    const uint4 v = row4[z];
                    rk += (v.x < key ? 1 : 0) + (v.y < key ? 1 : 0) + (v.z < key ? 1 : 0) + (v.w < key ? 1 : 0);
                }
                int v = (int)((key >> 5) | ((key & 31u) << kCodeShift));
                int lim = mrow;
                if (t - f >= have) {             // padding
                    rk = t - f;
                    v = ia;
                    lim = b.nbr_il ? (mrow + 3) & ~3 : 0;
                }
                if (rk < lim) {
                    if (b.nbr_il) b.nbr[((size_t)(rk >> 2) * b.ntot + ia) * 4 + (rk & 3)] = v;
                    else b.nbr[(size_t)ia * cap + rk] = v;
                }
            }
        }
        if (lane < mh) {
            const int ia = unpack_index(sh.home[lane].w);
            b.cnt[ia] = cnt;
            if (cnt > cap) atomicOr(&st.err, NEFE_ERR_NBR_OVERFLOW);
        }
        __syncwarp();                            // the home table and key rows are reused
    }
}

// Each warp takes a contiguous range of the worklist cells: with a worklist, the cells of the
// flagged systems in system order (rcbase[s] = first worklist cell of system s, rcbase[nsys] =
// their number); without one (stateless calls, one system), every cell of system 0.
template <typename F>
__device__ __forceinline__ void for_cells_of_grid(const Bufs& b, int nsys, F&& body) {
    const int nw = gridDim.x * (kTile / 32);
    const int wid = blockIdx.x * (kTile / 32) + (int)(threadIdx.x >> 5);
    if (b.by_flag) {                             // few systems: lane s holds the cells up to those of system s
        if (*(volatile int*)b.any_rebuild == 0) return;
        const int lane = threadIdx.x & 31;
        int upto = 0;
        if (lane < nsys) {
            const DevState& st = b.st[lane];
            if (st.rebuild) upto = st.ncell[0] * st.ncell[1] * st.ncell[2];
        }
        const int own = upto;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(0xffffffffu, upto, o);
            if (lane >= o) upto += y;
        }
        const int C = __shfl_sync(0xffffffffu, upto, 31), K = (C + nw - 1) / nw;
        const int g1 = min(C, (wid + 1) * K);
        for (int g = wid * K; g < g1; ++g) {
            const int s = __popc(__ballot_sync(0xffffffffu, upto <= g));
            body(s, g - __shfl_sync(0xffffffffu, upto - own, s));
        }
        return;
    }
    int C;
    if (b.rcbase) {
        C = b.rcbase[nsys];
    } else {
        const DevState& s0 = b.st[0];
        C = s0.ncell[0] * s0.ncell[1] * s0.ncell[2];
    }
    const int K = (C + nw - 1) / nw;
    const int g0 = wid * K, g1 = min(C, g0 + K);
    if (g0 >= g1) return;
    int s = 0;
    if (b.rcbase) {                              // largest s with rcbase[s] <= g0
        int lo = 0, hi = nsys;
        while (hi - lo > 1) {
            const int mid = (lo + hi) >> 1;
            if (b.rcbase[mid] <= g0) lo = mid; else hi = mid;
        }
        s = lo;
    }
    for (int g = g0; g < g1; ++g) {
        if (b.rcbase) {
            while (s + 1 < nsys && b.rcbase[s + 1] <= g) ++s;
        }
        body(s, g - (b.rcbase ? b.rcbase[s] : 0));
    }
}

template <typename T>
__device__ void nlist_cells_of_grid(const Bufs& b, int nsys, CellListShared<T>* shm) {
    const int lane = threadIdx.x & 31;
    CellListShared<T>& sh = shm[threadIdx.x >> 5];
    for_cells_of_grid(b, nsys, [&](int s, int c) { nlist_cell<T>(b, s, c, sh, lane); });
}

template <typename T>
__global__ void __launch_bounds__(kTile, 8) k_nlist_cell(Bufs b, int nsys) {
    dep_wait();
    __shared__ CellListShared<T> shm[kTile / 32];
    nlist_cells_of_grid<T>(b, nsys, shm);
}

// ------------------------------------------------------------------------------------
// The engine's whole rebuild in one cooperative launch (all blocks resident): worklist (block
// 0), cell count, scan, fill and list build, separated by grid barriers.  On a step where no list
// is stale every block returns at once, so the step pays one near-empty launch instead of five.
//
// Grid barrier: one 32-bit word; block 0 adds 2^31 - (nblocks - 1), every other block adds 1, so
// the word's top bit flips exactly when the last block arrives and its low bits return to what
// they were (the word needs no reset between barriers or launches).  Each block waits for the
// top bit it saw to flip, for at most kBarrierNs of %globaltimer; a block that gives up sets the
// context's timeout word and NEFE_ERR_TIMEOUT in every system and returns (the host then reports
// NEFE_ETIMEOUT and resets the words).  The launch is cooperative, so the wait never depends on a
// block that is not resident.
// ------------------------------------------------------------------------------------
constexpr unsigned long long kBarrierNs = 1000000000ULL;   // 1 s

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Returns false (in every thread of the block) when the wait gave up.
__device__ bool grid_barrier(unsigned* word, int* timeout, unsigned long long limit_ns, unsigned nblocks) {
    __shared__ int s_ok;
    __syncthreads();
    if (threadIdx.x == 0) {
        const unsigned add = blockIdx.x == 0 ? 0x80000000u - (nblocks - 1u) : 1u;
        __threadfence();
        const unsigned old = atomicAdd(word, add);
        int ok = 1;
        const unsigned long long t0 = global_ns();
        while (((*(volatile unsigned*)word ^ old) & 0x80000000u) == 0u) {
            if (global_ns() - t0 > limit_ns) {
                ok = 0;
                atomicOr(timeout, 1);
                break;
            }
            __nanosleep(64);
        }
        __threadfence();
        s_ok = ok;
    }
    __syncthreads();
    return s_ok != 0;
}

__device__ void flag_timeout(const Bufs& b, int nsys) {
    for (int s = threadIdx.x; s < nsys; s += blockDim.x) atomicOr(&b.st[s].err, NEFE_ERR_TIMEOUT);
}

template <typename T>
__global__ void __launch_bounds__(kTile, 8) k_rebuild_coop(Bufs b, int nsys) {
    __shared__ CellListShared<T> shm[kTile / 32];
    // no flag set anywhere this step: the word is written only by the kernels before this one
    if (*(volatile int*)b.any_rebuild == 0) {
        if (blockIdx.x == 0 && threadIdx.x == 0) {
            *b.rcount = 0;
            b.rcbase[nsys] = 0;
        }
        return;
    }
    unsigned* bar = reinterpret_cast<unsigned*>(b.any_rebuild + 3);
    int* tmo = b.any_rebuild + 2;
    const unsigned nb = gridDim.x;
    if (blockIdx.x == 0) build_worklist(b, nsys, 0);
    if (!grid_barrier(bar, tmo, kBarrierNs, nb)) { flag_timeout(b, nsys); return; }
    NEFE_FOR_TILES(b, cells_count_tile<T>(b, tile, threadIdx.x));
    if (!grid_barrier(bar, tmo, kBarrierNs, nb)) { flag_timeout(b, nsys); return; }
    for (int sy = blockIdx.x; sy < nsys; sy += gridDim.x)
        if (b.st[sy].rebuild) scan_system_cells(b, sy);
    if (!grid_barrier(bar, tmo, kBarrierNs, nb)) { flag_timeout(b, nsys); return; }
    NEFE_FOR_TILES(b, cells_fill_tile<T>(b, tile, threadIdx.x));
    if (!grid_barrier(bar, tmo, kBarrierNs, nb)) { flag_timeout(b, nsys); return; }
    nlist_cells_of_grid<T>(b, nsys, shm);
}

// Test of the barrier's time limit: a grid whose barrier expects one block more than it has
// (nothing will ever complete it), with a short limit; every block gives up and sets *timeout.
__global__ void __launch_bounds__(kTile) k_barrier_selftest(unsigned* word, int* timeout, unsigned long long ns) {
    grid_barrier(word, timeout, ns, gridDim.x + 1u);
}

// ------------------------------------------------------------------------------------
// Uhlenbeck-Ford fluid (the liquid's reference system, Sec. 2.1):
//   u(r) = -p kT ln(1 - exp(-r^2/sigma^2)) - u(rc),  r < rc.
// R6 (rebuild): UF pair rows, one warp per cell as in R5: the atoms of a cell share the 125 cells
// o in {-2..2}^3 around it (cells are at least rcs wide and rc + skin <= 2 rcs, so they cover the list
// radius; with at least 5 cells per axis no cell is visited twice).  Lane r < 25 looks up x-run r, one
// piece or two where it wraps at the box edge; the warp then walks the runs' candidates as one
// sequence, 32 at a time, and every candidate is tested against each atom of the cell (up to kUfHome
// at a time): j is appended when it lies within the list radius (rc + skin, mirror distance with a
// relative margin of 1e-5: the list only has to contain every pair that can come within rc before the
// next rebuild).  Rows are in cell order, not sorted: the force kernel sums in fixed point, so the
// order does not matter.  Bound by load latency: one thread per atom took its 490 candidates one after
// the other, 4 x 8000 atoms 57 us averaged over the steps -> 10.5 us.
// ------------------------------------------------------------------------------------
constexpr int kUfHome = 16;              // cell atoms per walk
constexpr int kUfPieces = 50;            // two per run (the second empty unless the run wraps)
template <typename T>
struct UfListShared {
    using T4 = typename V4<T>::t;
    T4 home[kUfHome];
    int4 edge[kUfPieces];                // first candidate of the piece's 2nd .. 5th cell
    int4 info[kUfPieces];                // first candidate, first flat index, code and x offset of the first cell
    int pw[kUfPieces];                   // first flat index again
};

template <typename T>
__device__ __forceinline__ void uflist_cell(const Bufs& b, int s, int c, UfListShared<T>& sh, int lane) {
    using T4 = typename V4<T>::t;
    constexpr unsigned kAll = 0xffffffffu;
    const DevSys& S = b.sys[s];
    if (S.uf_mode == UF_NONE) return;
    DevState& st = b.st[s];
    const int* start = b.cell_start + S.cell0 + s;
    const int n = S.n, off = S.off;
    const int hs = max(0, min(start[c], n)), m = max(hs, min(start[c + 1], n)) - hs;
    if (m == 0) return;
    const T4* xc = reinterpret_cast<const T4*>(b.xcs) + off;
    const int nx = st.ncell[0], ny = st.ncell[1], nz = st.ncell[2];
    if (nx < 5 || ny < 5 || nz < 5) {
        for (int q = lane; q < m; q += 32) {
            const int i = unpack_index(xc[hs + q].w);
            if ((unsigned)(i - off) < (unsigned)n) b.uf_cnt[i] = 0;
        }
        atomicOr(&st.err, NEFE_ERR_BOX);
        return;
    }
    const T hx = pick<T>(st.h[0], st.h_f[0]), hy = pick<T>(st.h[1], st.h_f[1]), hz = pick<T>(st.h[2], st.h_f[2]);
    const T R2 = pick<T>(S.uf_R2 * (1.0 + 1e-5), S.uf_R2_f * (1.0f + 1e-5f));
    const int cx = c % nx, cy = (c / nx) % ny, cz = c / (nx * ny);
    // run r = (oy, oz): cells cx - 2 .. cx + 2 as piece A = ox < brk and piece B = the rest, past the edge
    const int brk = cx < 2 ? -cx : (cx + 2 >= nx ? nx - cx : 3);
    const int na = brk + 2, nb = 3 - brk;
    const int xa = cx < 2 ? cx - 2 + nx : cx - 2;
    int pa[6], pb[6];                            // starts of the cells of each piece, then its end
    int len = 0;
    if (lane < 25) {
        int yy = cy + lane % 5 - 2, zz = cz + lane / 5 - 2;
        yy = yy < 0 ? yy + ny : (yy >= ny ? yy - ny : yy);
        zz = zz < 0 ? zz + nz : (zz >= nz ? zz - nz : zz);
        const int* row = start + nx * (yy + ny * zz);
#pragma unroll
        for (int k = 0; k < 6; ++k) {
            pa[k] = max(0, min(row[xa + min(k, na)], n));
            pb[k] = max(0, min(row[min(k, nb)], n));
        }
        len = max(0, pa[5] - pa[0]) + max(0, pb[5] - pb[0]);
    }
    int incl = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(kAll, incl, o);
        if (lane >= o) incl += y;
    }
    const int total = __shfl_sync(kAll, incl, 31);
    if (lane < 25) {
        const int f0 = incl - len, f1 = f0 + max(0, pa[5] - pa[0]);
        const int code = 5 * (lane % 5) + 25 * (lane / 5);
        sh.pw[2 * lane] = f0;
        sh.pw[2 * lane + 1] = f1;
        sh.edge[2 * lane] = make_int4(pa[1], pa[2], pa[3], pa[4]);
        sh.edge[2 * lane + 1] = make_int4(pb[1], pb[2], pb[3], pb[4]);
        sh.info[2 * lane] = make_int4(pa[0], f0, code, -2);
        sh.info[2 * lane + 1] = make_int4(pb[0], f1, code, brk);
    }
    for (int h0 = 0; h0 < m; h0 += kUfHome) {
        const int mh = min(kUfHome, m - h0);
        __syncwarp();
        if (lane < mh) sh.home[lane] = xc[hs + h0 + lane];
        __syncwarp();
        int cnt = 0;                             // lane a: entries of cell atom a
        for (int t0 = 0; t0 < total; t0 += 32) {
            const int t = t0 + lane;
            int j = -1, o = 0;
            // a candidate that is not one (past the sequence, or a bad index) sits far away
            T cxj = (T)1e15, cyj = (T)1e15, czj = (T)1e15;
            if (t < total) {
                int e = 0;                       // piece of t: last one whose flat start is <= t
#pragma unroll
                for (int step = 32; step > 0; step >>= 1) {
                    const int q = e + step;
                    if (q < kUfPieces && sh.pw[q] <= t) e = q;
                }
                const int4 in = sh.info[e], ed = sh.edge[e];
                const int p = in.x + (t - in.y);
                const T4 xj = xc[p];
                j = unpack_index(xj.w);
                const int ox = in.w + (p >= ed.x) + (p >= ed.y) + (p >= ed.z) + (p >= ed.w);
                o = in.z + ox + 2;
                if ((unsigned)(j - off) < (unsigned)n) {
                    cxj = xj.x + (T)ox * hx;
                    cyj = xj.y + (T)((e >> 1) % 5 - 2) * hy;
                    czj = xj.z + (T)((e >> 1) / 5 - 2) * hz;
                } else {
                    atomicOr(&st.err, NEFE_ERR_CELL);
                }
            }
            const unsigned ent = (unsigned)j | (unsigned)o << kUfShift;
            for (int a = 0; a < mh; ++a) {
                const T4 ha = sh.home[a];
                const int ia = unpack_index(ha.w);
                const T dx = cxj - ha.x, dy = cyj - ha.y, dz = czj - ha.z;
                const bool in = dx * dx + dy * dy + dz * dz < R2 && j != ia;
                const unsigned bal = __ballot_sync(kAll, in);
                const int pos = __shfl_sync(kAll, cnt, a) + __popc(bal & ((1u << lane) - 1u));
                if (in && pos < kUfCap && (unsigned)(ia - off) < (unsigned)n) b.uf_nbr[(size_t)ia * kUfCap + pos] = (int)ent;
                if (lane == a) cnt += __popc(bal);
            }
        }
        if (lane < mh) {
            const int ia = unpack_index(sh.home[lane].w);
            if ((unsigned)(ia - off) < (unsigned)n) b.uf_cnt[ia] = cnt;
            if (cnt > kUfCap) atomicOr(&st.err, NEFE_ERR_NBR_OVERFLOW);
        }
    }
    __syncwarp();                                // the tables are reused
}
template <typename T>
__global__ void __launch_bounds__(kTile) k_uflist(Bufs b, int nsys) {
    dep_wait();
    __shared__ UfListShared<T> shm[kTile / 32];
    UfListShared<T>& sh = shm[threadIdx.x >> 5];
    const int lane = threadIdx.x & 31;
    for_cells_of_grid(b, nsys, [&](int s, int c) { uflist_cell<T>(b, s, c, sh, lane); });
}

// Fixed-point accumulation of the UF pair sums (order independent, so the unsorted rows give
// bitwise reproducible forces): 2^-32 units in the FP32 kernel, 2^-40 in the FP64 kernel.
template <typename T> struct UfFix;
template <> struct UfFix<float> {
    __device__ static long long to(float v) { return __float2ll_rn(v * 4294967296.0f); }
    __device__ static float from(long long q) { return (float)((double)q * 0x1p-32); }
    __device__ static long long sum_unit(long long q) { return q; }                // to the sums' 2^-32
};
template <> struct UfFix<double> {
    __device__ static long long to(double v) { return __double2ll_rn(v * 0x1p40); }
    __device__ static double from(long long q) { return (double)q * 0x1p-40; }
    __device__ static long long sum_unit(long long q) { return (q + 128) >> 8; }
};

// A lane's sums.  FP32: a conversion to int64 runs on the FP64 pipe (it was 68 % busy with them), so
// round(v 2^32) is taken by two FP32 additions instead, for |v| < 64: v + 192 rounds v to 2^-16, the
// exact remainder plus 1.5 2^-9 rounds to 2^-32, and the bits of both less those of their constants are the
// integers, added as such.  The same integer as the conversion's, which larger values still take.
template <typename T, int K>
struct UfSum {
    long long q[K];
    __device__ __forceinline__ void clear(long long*) {
#pragma unroll
        for (int k = 0; k < K; ++k) q[k] = 0;
    }
    template <int M>
    __device__ __forceinline__ void add(const T (&v)[M], bool) {
#pragma unroll
        for (int k = 0; k < M; ++k) q[k] += UfFix<T>::to(v[k]);
    }
    __device__ __forceinline__ long long get(int k) const { return q[k]; }
};
template <int K>
struct UfSum<float, K> {
    int hi[K], lo[K];
    long long* q;                        // the larger values' sums: memory of the thread, hardly ever used
    bool any;
    __device__ __forceinline__ void clear(long long* local) {
#pragma unroll
        for (int k = 0; k < K; ++k) hi[k] = lo[k] = 0;
        q = local;
        any = false;
    }
    template <int M>
    __device__ __forceinline__ void add(const float (&v)[M], bool small) {
        if (__builtin_expect(small, 1)) {
            const float C = 192.0f, C2 = 0x1.8p-9f;
#pragma unroll
            for (int k = 0; k < M; ++k) {
                const float t = __fadd_rn(v[k], C);
                hi[k] += __float_as_int(t) - __float_as_int(C);
                lo[k] += __float_as_int(__fadd_rn(__fsub_rn(v[k], __fsub_rn(t, C)), C2)) - __float_as_int(C2);
            }
        } else {
            if (!any)
                for (int k = 0; k < K; ++k) q[k] = 0;
            any = true;
#pragma unroll 1
            for (int k = 0; k < M; ++k) q[k] += UfFix<float>::to(v[k]);
        }
    }
    __device__ __forceinline__ long long get(int k) const {
        return (any ? q[k] : 0LL) + (long long)hi[k] * 65536 + lo[k];
    }
};

// Energy u (without the shift) and force coefficient c (force on j along d: c d; on i: -c d) of a pair
// at xx = r^2/sigma^2: u = -pk ln(1 - e), c = (2 pk / sigma^2) e / (1 - e), e = exp(-xx).  FP32: from
// xx = 0.7 on, where 1 - e is at least one half, it is taken as it stands, and -ln(1 - e) = e + e^2 q(e)
// with q fitted (Chebyshev nodes, 8th degree) on [0, 1/2]: within 1.2e-7 of u, where ln of the rounded
// 1 - e loses the small e.
__device__ __forceinline__ void uf_pair(float xx, float pk, float c0, float& u, float& c) {
    const float e = expf(-xx);
    if (xx >= 0.7f) {
        constexpr float a[9] = {0x1.0p-1f, 0x1.555394p-2f, 0x1.0059eep-2f, 0x1.8bdac4p-3f, 0x1.da2ab2p-3f,
                                -0x1.9d06dcp-3f, 0x1.2944ccp+0f, -0x1.942780p+0f, 0x1.54cfd0p+0f};
        float q = a[8];
#pragma unroll
        for (int k = 7; k >= 0; --k) q = fmaf(q, e, a[k]);
        u = pk * fmaf(e * e, q, e);
        c = c0 * __fdividef(e, 1.0f - e);
    } else {
        const float m = -expm1f(-xx);
        u = -pk * logf(m);
        c = c0 * (e / m);
    }
}
__device__ __forceinline__ void uf_pair(double xx, double pk, double c0, double& u, double& c) {
    u = -pk * ::log(-::expm1(-xx));
    c = c0 / ::expm1(xx);
}

// Per step (or stateless): UF force and energy of each atom of a UF system from its row, kUfLanes
// lanes to an atom (the row read 32 bytes at a time; the fixed-point sums of the lanes add exactly).
// Each pair is seen from both ends: half its energy and virial per end, the full force.
// The energy goes to U_int (pot = UF) or to the FL reference energy U_E (UF reference); the
// virial enters the pressure only when the UF term is U_int.  FP32 distances come from fractional
// positions, FP64 ones from the mirror and the entry's cell offset.
// One thread per atom left most of the chip idle (142 entries one after the other, each lane in a row
// of its own): 4 x 8000 atoms 155 -> 34 us.
// (FP64 keeps a tile to a block: its block sums are rounded to 2^-32 once per 128 atoms.)
template <typename T> constexpr int kUfLanes = sizeof(T) == 8 ? 4 : 8;
template <typename T> constexpr int kUfThreads = sizeof(T) == 8 ? 4 * kTile : kTile;
template <typename T> constexpr int kUfBlocks = kTile * kUfLanes<T> / kUfThreads<T>;   // per tile
template <typename T, int MODE, bool FINE>
__global__ void __launch_bounds__(kUfThreads<T>, sizeof(T) == 4 ? 5 : 1) k_uf(Bufs b) {
    dep_wait();
    using T4 = typename V4<T>::t;
    constexpr bool kFrac = sizeof(T) == 4;
    constexpr int L = kUfLanes<T>, PARTS = kUfBlocks<T>, G = kTile / PARTS;   // atoms per block
    __shared__ T4 soff[kFrac ? 1 : 125];
    const int item = (int)blockIdx.x / PARTS, part = (int)blockIdx.x % PARTS;
    const TileAtom ta = tile_of(b, b.uf_tiles ? b.uf_tiles[item] : item);
    const DevSys& S = b.sys[ta.sys];
    DevState& st = b.st[ta.sys];
    if (S.uf_mode == UF_NONE) return;            // uniform over the block
    const bool pressure = S.uf_mode == UF_INT;
    if constexpr (!kFrac) {
        if (threadIdx.x < 125) {
            const int c = threadIdx.x;
            soff[c] = mk4((T)(c % 5 - 2) * (T)st.h[0], (T)((c / 5) % 5 - 2) * (T)st.h[1], (T)(c / 25 - 2) * (T)st.h[2], (T)0);
        }
        __syncthreads();
    }
    const T pk = pick<T>(S.uf_pk, S.uf_pk_f), is2 = pick<T>(S.uf_is2, S.uf_is2_f);
    const T rc2 = pick<T>(S.uf_rc2, S.uf_rc2_f), shift = pick<T>(S.uf_shift, S.uf_shift_f);
    const T c0 = (T)2 * pk * is2;
    const T cmax = (T)64 / fmax(sqrt(rc2), (T)0.5 * rc2);   // below it no term reaches 64
    UfSum<T, 10> sum;                            // f xyz, energy, virial xx yy zz xy xz yz
    long long large[kFrac ? 10 : 1];
    sum.clear(large);
    const int lane = threadIdx.x % L, ia = part * G + (int)threadIdx.x / L;
    const bool valid = ia < ta.count;
    const int i = ta.first + ia;
    if (valid) {
        const int cnt = min(b.uf_cnt[i], kUfCap);
        const int* row = b.uf_nbr + (size_t)i * kUfCap;
        int4 fi = make_int4(0, 0, 0, 0);
        T4 xi = mk4((T)0, (T)0, (T)0, (T)0);
        float4 Lh = make_float4(0.f, 0.f, 0.f, 0.f), Ll = Lh;
        if constexpr (kFrac) {
            fi = b.xf[i];
            Lh = b.lscale[4 * ta.sys];
            Ll = b.lscale[4 * ta.sys + 1];
        } else {
            xi = reinterpret_cast<const T4*>(b.xs)[i];
        }
        // the entry two turns ahead and the position one turn ahead are loaded before a turn's arithmetic
        const int last = cnt - 1;
        auto entry = [&](int a) { return (unsigned)row[min(a, last)]; };
        using P4 = std::conditional_t<kFrac, int4, T4>;
        auto position = [&](unsigned e) {
            const int j = (e & kUfMask) < (unsigned)b.ntot ? (int)(e & kUfMask) : i;
            if constexpr (kFrac) return b.xf[j];
            else return reinterpret_cast<const T4*>(b.xs)[j];
        };
        unsigned e1 = 0u, e2 = 0u;
        P4 p1{};
        if (lane < cnt) {
            e1 = entry(lane);
            e2 = entry(lane + L);
            p1 = position(e1);
        }
        for (int a = lane; a < cnt; a += L) {
            const unsigned e = e1;
            const P4 xj = p1;
            e1 = e2;
            e2 = entry(a + 2 * L);
            p1 = position(e1);
            if (!NEFE_IN_RANGE(e & kUfMask, b.ntot, &st.err)) continue;
            T dx, dy, dz;
            if constexpr (kFrac) {
                float gx = (float)wrap_sub(xj.x, fi.x), gy = (float)wrap_sub(xj.y, fi.y), gz = (float)wrap_sub(xj.z, fi.z);
                if constexpr (FINE) {
                    const float3 g = frac_low_diff(xj.w, fi.w);
                    gx += g.x; gy += g.y; gz += g.z;
                }
                dx = gx * Lh.x + gx * Ll.x; dy = gy * Lh.y + gy * Ll.y; dz = gz * Lh.z + gz * Ll.z;
            } else {
                const T4 oh = soff[e >> kUfShift];
                dx = (xj.x - xi.x) + oh.x; dy = (xj.y - xi.y) + oh.y; dz = (xj.z - xi.z) + oh.z;
            }
            const T r2 = dx * dx + dy * dy + dz * dz;
            if (!(r2 < rc2)) continue;
            T u, c;
            uf_pair(r2 * is2, pk, c0, u, c);
            const bool small = c < cmax && u < (T)64;
            const T hc = (T)0.5 * c, eh = (T)0.5 * (u - shift);
            if (pressure) sum.add({-c * dx, -c * dy, -c * dz, eh, hc * dx * dx, hc * dy * dy, hc * dz * dz, hc * dx * dy, hc * dx * dz, hc * dy * dz}, small);
            else sum.add({-c * dx, -c * dy, -c * dz, eh}, small);
        }
    }
    long long q[10];
#pragma unroll
    for (int k = 0; k < 10; ++k) q[k] = sum.get(k);
    // the atom's sums, then (lanes of different atoms) the warp's.  An atom whose energy or virial left
    // the range (a pair at zero distance saturates) is reported, and kept out of the block's sums.
#pragma unroll
    for (int k = 0; k < 10; ++k) {
        if (k > 3 && !pressure) break;           // (uniform)
#pragma unroll
        for (int o = L / 2; o > 0; o >>= 1) q[k] += __shfl_xor_sync(0xffffffffu, q[k], o);
    }
    if (valid && lane == 0) {
        T v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) v[k] = UfFix<T>::from(q[k]);
        if (MODE == FM_FORCES) {
            const size_t N = b.ntot;
            b.f_out[i] = (double)v[0]; b.f_out[N + i] = (double)v[1]; b.f_out[2 * N + i] = (double)v[2];
            if (b.e_atom) b.e_atom[i] = (double)v[3];
        } else {
            reinterpret_cast<T4*>(b.uf_F)[i] = mk4(v[0], v[1], v[2], v[3]);
        }
    }
    bool out = false;
#pragma unroll
    for (int k = 3; k < 10; ++k) {
        const long long x = UfFix<T>::sum_unit(q[k]);
        out = out || x >= (1LL << 47) || x <= -(1LL << 47);
    }
    if (out) atomicOr(&st.err, NEFE_ERR_NAN);
    __shared__ long long red[kUfThreads<T> / 32][7];     // energy, virial
#pragma unroll
    for (int k = 0; k < 7; ++k) {
        long long x = out ? 0 : q[3 + k];
#pragma unroll
        for (int o = 16; o >= L; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5][k] = x;
    }
    __syncthreads();
    if (threadIdx.x < (pressure ? 7 : 1)) {
        const int k = threadIdx.x;
        long long x = 0;
        for (int w = 0; w < kUfThreads<T> / 32; ++w) x += red[w][k];
        x = UfFix<T>::sum_unit(x);
        if (x >= (1LL << 47) || x <= -(1LL << 47)) {
            atomicOr(&st.err, NEFE_ERR_NAN);
        } else if (x != 0) {
            const int slot = !pressure ? ACC_UREF : k == 0 ? ACC_UINT : ACC_VIR + k - 1;
            atomicAdd(reinterpret_cast<unsigned long long*>(
                          &b.acc[((size_t)ta.sys * ACC_N + slot) * kSlots + (blockIdx.x % kSlots)]),
                      (unsigned long long)x);
        }
    }
}

// Mirror only (stateless forces): same q / xs formula as R1, without counting.
template <typename T>
__global__ void __launch_bounds__(kTile) k_mirror(Bufs b) {
    dep_wait();
    using T4 = typename V4<T>::t;
    const TileAtom ta = tile_of(b, blockIdx.x);
    const DevState& st = b.st[ta.sys];
    if ((int)threadIdx.x >= ta.count) return;
    const int i = ta.first + threadIdx.x;
    double xs[3];
    for (int k = 0; k < 3; ++k) {
        const double xk = b.x[(size_t)k * b.ntot + i];
        int q, c;
        cell_axis(xk, st.box[k], st.ibox[k] * (double)st.ncell[k], st.ncell[k], q, c);
        xs[k] = xk - (double)q * st.h[k];
    }
    reinterpret_cast<T4*>(b.xs)[i] = mk4((T)xs[0], (T)xs[1], (T)xs[2], (T)0);
    if (b.xc) {
        const size_t N = b.ntot;
        const double x3[3] = {b.x[i], b.x[N + i], b.x[2 * N + i]};
        b.xc[i] = pack_frac(frac_position(x3, st, 0));
        if (i == 0) scale_of_box(b, 0, st);
    }
}

// ------------------------------------------------------------------------------------
// Half kick + drift.  mode 0 (setup): mirror and noise only.
// x = anchor + dhi + dlo; per step the displacement grows by dt phi v + (s - 1) x (affine
// box drift).  In the FP32 path (dhi, dlo) is a compensated pair: a two-sum keeps the
// rounding error of every increment in dlo.
// ------------------------------------------------------------------------------------
// Every operation is rounded by itself (no contraction with the product that made d), so that the
// two kernels that move atoms give the same bits whatever surrounds the call in each.
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ float fma_rn(float a, float b, float c) { return __fmaf_rn(a, b, c); }
__device__ __forceinline__ double fma_rn(double a, double b, double c) { return __fma_rn(a, b, c); }
template <typename T>
__device__ __forceinline__ void comp_add(T& hi, T& lo, T d) {
    if constexpr (sizeof(T) == 8) {
        hi = __dadd_rn(hi, d);
    } else {
        const T s = __fadd_rn(hi, d);
        const T bp = __fsub_rn(s, hi);
        const T err = __fadd_rn(__fsub_rn(hi, __fsub_rn(s, bp)), __fsub_rn(d, bp));
        lo = __fadd_rn(lo, err);
        const T h2 = __fadd_rn(s, lo);
        lo = __fsub_rn(lo, __fsub_rn(h2, s));
        hi = h2;
    }
}

// Constants of the fractional positions' update (rows 2 and 3 of lscale).
struct BoxMove {
    float omr[3], to_frac[3];
};
__device__ __forceinline__ BoxMove box_move(const Bufs& b, int s) {
    const float4 o = b.lscale[4 * s + 2], t = b.lscale[4 * s + 3];
    return {{o.x, o.y, o.z}, {t.x, t.y, t.z}};
}

// Position of atom i from its displacement d since the last build: the mirror (want_xs) and, in the
// FP32 path, the fractional position (want_xf), which the scatter form's pass A reads.  Returns the
// squared displacement of the list test, relative to the box's own deformation.  With x = X + d (X at
// the build) and the cell edge grown from hb to h, the fraction is X/L_b + [d + X (1 - h/hb)] / L.
template <typename T>
__device__ __forceinline__ T place_atom(const Bufs& b, const DevState& st, const BoxMove& bm, int i,
                                        const typename V4<T>::t& xa, const int4& fb, const int4& q, const T (&d)[3]) {
    using T4 = typename V4<T>::t;
    const T xav[3] = {xa.x, xa.y, xa.z};
    const int qa[3] = {q.x, q.y, q.z};
    const bool hmoved = st.hmoved != 0;
    T dd2 = 0;
    if constexpr (sizeof(T) == 8) {
        T m[3];
        for (int k = 0; k < 3; ++k) {
            m[k] = xav[k] + d[k];
            if (hmoved) m[k] -= (T)qa[k] * (st.h[k] - st.hb[k]);
            const T dd = hmoved ? m[k] - xav[k] * (st.h[k] / st.hb[k]) : d[k];
            dd2 += dd * dd;
        }
        reinterpret_cast<T4*>(b.xs)[i] = mk4(m[0], m[1], m[2], (T)0);
        if (b.want_xf) {                         // the row filter's position (FP32 does for it)
            float mv[3];
            for (int k = 0; k < 3; ++k) {
                mv[k] = (float)d[k];
                if (hmoved) mv[k] = fmaf(fmaf((float)qa[k], st.hb_f[k], (float)xav[k]), bm.omr[k], mv[k]);
            }
            b.xc[i] = pack_frac(frac_moved(fb, mv[0] * bm.to_frac[0], mv[1] * bm.to_frac[1], mv[2] * bm.to_frac[2], 0));
        }
    } else {
        T mv[3];
        for (int k = 0; k < 3; ++k) {
            mv[k] = d[k];
            // (the list test alone does with the FP32 ratio)
            if (hmoved) mv[k] = fma_rn(fma_rn((T)qa[k], st.hb_f[k], xav[k]), b.want_xf ? bm.omr[k] : 1.0f - st.rho_f[k], mv[k]);
            dd2 += mv[k] * mv[k];
        }
        if (b.want_xf) {
            const int4 f = frac_moved(fb, mul_rn(mv[0], bm.to_frac[0]), mul_rn(mv[1], bm.to_frac[1]),
                                      mul_rn(mv[2], bm.to_frac[2]), b.want_xf > 1);
            b.xf[i] = f;
            b.xc[i] = pack_frac(f);
        }
        if (b.want_xs) {
            T m[3];
            for (int k = 0; k < 3; ++k) {
                m[k] = xav[k] + d[k];
                if (hmoved) m[k] -= (T)qa[k] * (st.h_f[k] - st.hb_f[k]);
            }
            reinterpret_cast<T4*>(b.xs)[i] = mk4(m[0], m[1], m[2], (T)0);
        }
    }
    return dd2;
}

// Drift of atom i by its half-kicked velocity vk (move), its position (place_atom), the
// displacement test (sets *flag) and the thermostat noise of step kstep (stored, and returned in
// z).  dh, dl: the atom's displacement, updated in place.  Shared by k_kick_drift and by the epilogue
// that moves the atoms for the next step (systems without a barostat), so both do the same
// operations.  xa, fb: the atom's mirror and fractional position at the last build (loaded by the
// caller together with its other operands).  any: the context-wide word that records that some system's flag was set (or NULL).
template <typename T>
__device__ __forceinline__ void drift_atom(const Bufs& b, const DevSys& S, const DevState& st, const BoxMove& bm, int i,
                                           const typename V4<T>::t& xa, const int4& fb, const T (&vk)[3], bool move,
                                           T (&dh)[3], T (&dl)[3], int flag_set, int* flag, int* any,
                                           unsigned long long kstep, T (&z)[3],
                                           const typename V4<T>::t* drawn = nullptr) {
    using T4 = typename V4<T>::t;
    const size_t N = b.ntot;
    T* DH = reinterpret_cast<T*>(b.dhi);
    T* DL = reinterpret_cast<T*>(b.dlo);
    const T xav[3] = {xa.x, xa.y, xa.z};
    const bool scaled = st.scaled != 0, hmoved = st.hmoved != 0;
    int4 q = make_int4(0, 0, 0, 0);
    if (scaled || hmoved) q = b.q[i];
    const int qa[3] = {q.x, q.y, q.z};
    if (move) {
        const T dt = pick<T>(b.dt, S.dt_f);
        for (int k = 0; k < 3; ++k) {
            T d = mul_rn(mul_rn(dt, pick<T>(st.phi[k], st.phi_f[k])), vk[k]);
            if (scaled) {   // (s - 1) x with x = xa + q hb + displacement
                const T xk = fma_rn((T)qa[k], pick<T>(st.hb[k], st.hb_f[k]), xav[k]) + dh[k];
                d = fma_rn(pick<T>(st.s[k] - 1.0, st.sm1_f[k]), xk, d);
            }
            comp_add<T>(dh[k], dl[k], d);
            DH[k * N + i] = dh[k];
            if constexpr (sizeof(T) == 4) DL[k * N + i] = dl[k];
        }
    }
    const T d[3] = {dh[0] + dl[0], dh[1] + dl[1], dh[2] + dl[2]};
    const T dd2 = place_atom<T>(b, st, bm, i, xa, fb, q, d);
    if (dd2 > pick<T>(st.thr2, st.thr2_f) && !flag_set) {
        atomicOr(flag, 1);
        if (any) atomicOr(any, 1);
    }
    z[0] = z[1] = z[2] = (T)0;
    if (S.thermo) {
        if (drawn) {
            z[0] = drawn->x; z[1] = drawn->y; z[2] = drawn->z;
        } else {
            Noise<T>::xi3(S.seed, (uint64_t)S.rng_id, (uint64_t)kstep, (uint64_t)(i - S.off), z);
        }
        reinterpret_cast<T4*>(b.xi)[i] = mk4(z[0], z[1], z[2], (T)0);
    }
}

// Positions of every atom from the anchor and the displacement, in the forms that the force passes
// in use read (after a checkpoint was loaded or another form was chosen).
template <typename T>
__global__ void __launch_bounds__(kTile) k_positions(Bufs b) {
    dep_wait();
    using T4 = typename V4<T>::t;
    __shared__ BoxMove bm;
    const TileAtom ta = tile_of(b, blockIdx.x);
    const DevState& st = b.st[ta.sys];
    if (threadIdx.x < 3) {                       // (the rows of lscale are written below)
        const int k = threadIdx.x;
        bm.omr[k] = st.hmoved ? (float)(1.0 - st.h[k] / st.hb[k]) : 0.0f;
        bm.to_frac[k] = 4294967296.0f / (float)st.box[k];
    }
    __syncthreads();
    if ((int)threadIdx.x >= ta.count) return;
    const int i = ta.first + threadIdx.x;
    const size_t N = b.ntot;
    if (b.want_xf && i == b.sys[ta.sys].off) scale_of_box(b, ta.sys, st);
    int4 fb = make_int4(0, 0, 0, 0);
    if (b.want_xf) {
        const double x[3] = {b.x[i], b.x[N + i], b.x[2 * N + i]};
        b.xfb[i] = fb = frac_position(x, st, b.want_xf > 1);
    }
    T d[3];
    for (int k = 0; k < 3; ++k) {
        d[k] = reinterpret_cast<const T*>(b.dhi)[k * N + i];
        if constexpr (sizeof(T) == 4) d[k] += reinterpret_cast<const T*>(b.dlo)[k * N + i];
    }
    place_atom<T>(b, st, bm, i, reinterpret_cast<const T4*>(b.xa)[i], fb, b.q[i], d);
}

// drawn: the step's noise is in xi_next (draw_ahead).
// skip: systems without a barostat were already kicked and moved by the previous step's
// epilogue (k_finish with fuse), so their tiles return at once.
template <typename T>
__global__ void __launch_bounds__(kTile) k_kick_drift(Bufs b, int mode, int skip, int drawn) {
    dep_wait();
    using T4 = typename V4<T>::t;
    const TileAtom ta = tile_of(b, blockIdx.x);
    const DevSys& S = b.sys[ta.sys];
    DevState& st = b.st[ta.sys];
    if (skip && S.baro == BARO_NONE) return;     // uniform over the block (one system per tile)
    const BoxMove bm = b.want_xf ? box_move(b, ta.sys) : BoxMove{};
    T xs_sum[3] = {(T)0, (T)0, (T)0};
    if ((int)threadIdx.x < ta.count) {
        const int i = ta.first + threadIdx.x;
        const size_t N = b.ntot;
        T* V = reinterpret_cast<T*>(b.v);
        const T* DH = reinterpret_cast<const T*>(b.dhi);
        const T* DL = reinterpret_cast<const T*>(b.dlo);
        const T4 xa = reinterpret_cast<const T4*>(b.xa)[i];
        int4 fb = make_int4(0, 0, 0, 0);
        if (b.want_xf) fb = b.xfb[i];
        T dh[3], dl[3], vk[3] = {(T)0, (T)0, (T)0};
        for (int k = 0; k < 3; ++k) {
            dh[k] = DH[k * N + i];
            if constexpr (sizeof(T) == 4) dl[k] = DL[k * N + i]; else dl[k] = (T)0;
        }
        if (mode == 1) {
            const T4 F = reinterpret_cast<const T4*>(b.F)[i];
            const T fv[3] = {F.x, F.y, F.z};
            const T ck = pick<T>(S.ckick, S.ckick_f);
            for (int k = 0; k < 3; ++k) {
                vk[k] = fma_rn(ck, fv[k], V[k * N + i]);
                V[k * N + i] = vk[k];
            }
        }
        drift_atom<T>(b, S, st, bm, i, xa, fb, vk, mode == 1, dh, dl, st.rebuild, &st.rebuild, b.any_rebuild,
                      (unsigned long long)st.k,
                      xs_sum, drawn ? reinterpret_cast<const T4*>(b.xi_next) + i : nullptr);
    }
    block_sum_to_acc<T, 3>(xs_sum, b.acc + (size_t)ta.sys * ACC_N * kSlots, ACC_XI, &st.err);
}

// ------------------------------------------------------------------------------------
// Stillinger-Weber terms for one edge of length r (A):
//   phi = eps A (B s^-p - s^-q) exp(1/(s - a)),  g = exp(gamma/(s - a)),  s = r/sigma,
// with dphi/dr and dg/dr.
// ------------------------------------------------------------------------------------
// Distance (in sigma) below the cutoff a inside which an edge is treated as cut off: there
// exp(1/(s - a)) and exp(gamma/(s - a)) underflow to 0 anyway, and 1/(s - a) would overflow
// (0 * inf = NaN) when s rounds onto a.
template <typename T> __device__ __forceinline__ T cut_eps() { return sizeof(T) == 4 ? (T)1e-5 : (T)1e-12; }

template <typename T>
__device__ __forceinline__ void sw_edge(const SWc<T>& P, T r, T& phi, T& dphi, T& g, T& dg) {
    const T s = r * P.inv_sig;
    if (!(s < P.s_act) || !(s - P.a < -cut_eps<T>())) {
        phi = dphi = g = dg = (T)0;
        return;
    }
    const T id = xrcp(s - P.a);
    const T e1 = xexp(id);
    g = xexp(P.gam * id);
    T rp, rq;
    if (P.int_pq) {
        const T is2 = xrcp(s * s);
        rp = is2 * is2;
        rq = (T)1;
    } else {
        rp = xpow(s, -P.p);
        rq = xpow(s, -P.q);
    }
    const T poly = P.B * rp - rq;
    phi = P.epsA * poly * e1;
    dphi = P.epsA * e1 * ((-P.p * P.B * rp + P.q * rq) * xrcp(s) - poly * id * id) * P.inv_sig;
    dg = -g * P.gam * id * id * P.inv_sig;
}

// Derivatives of one pair term phi2(r) with respect to A, B, p, q, a (sigma, eps fixed):
// phi2 = eps A (B s^-p - s^-q) e,  e = exp(1/(s - a)).
template <typename T>
__device__ __forceinline__ void sw_pair_pgrad(const SWc<T>& P, T r, T out[5]) {
    const T s = r * P.inv_sig;
    if (!(s < P.s_act) || !(s - P.a < -cut_eps<T>())) {
        for (int k = 0; k < 5; ++k) out[k] = (T)0;
        return;
    }
    const T id = xrcp(s - P.a);
    const T e1 = xexp(id);
    const T ls = xlog(s);
    const T rp = xpow(s, -P.p), rq = xpow(s, -P.q);
    const T ea = P.eps * P.A * e1;
    const T phi = ea * (P.B * rp - rq);
    out[0] = phi / P.A;                 // d/dA
    out[1] = ea * rp;                   // d/dB
    out[2] = -ea * P.B * rp * ls;       // d/dp
    out[3] = ea * rq * ls;              // d/dq
    out[4] = phi * id * id;             // d/da (pair exponent)
}

// Force pass A.  L lanes per atom, 128/L atoms per block.
//  1. The lanes compact the atom's Verlet row into its in-cutoff shell: (d, r^2) in shared
//     memory, the neighbour indices in shj (ended by -1 when shorter than kShell).
//  2. Lane a owns shell edge a: pair term (full force on i, half the energy), g, dg/dr and the
//     unit vector u_a.
//  3. Lane a sums over the other edges b the force that triplet (i; a, b) exerts on the leg
//     atom j_a,  F_a(b) = -t1 u_b + (t1 c - t2) u_a  with  c = u_a.u_b,
//     t1 = 2 eps lambda (c - c0) g_a g_b / r_a,  t2 = eps lambda (c - c0)^2 g_b (dg/dr)_a,
//     and stores the leg force L_a = sum_b F_a(b) in shd[i][a] for pass B.  Atom i gets -L_a
//     (the three forces of a triplet sum to zero) and half of h(i; a, b) per ordered pair.
// Each ordered pair costs ~14 flops and every triplet force is computed exactly once.
// P[i] = (pair + own triplet force, atom energy), then the atom's virial.
template <typename T, int L>
__global__ void __launch_bounds__(kTile) k_edges(Bufs b) {
    dep_wait();
    using T4 = typename V4<T>::t;
    constexpr int G = kTile / L;
    // rows padded by one entry: the groups of a warp then start on different banks
    __shared__ T4 sh_u[G][kShell + 1];     // (d, r^2) after compaction, then (u, r)
    __shared__ T sh_g[G][kShell + 1];
    __shared__ T sh_dg[G][kShell + 1];
    __shared__ T4 soff[27];

    const int tile = blockIdx.x / L + b.tile_base, part = blockIdx.x % L;
    const TileAtom ta = tile_of(b, tile);
    const DevSys& S = b.sys[ta.sys];
    DevState& st = b.st[ta.sys];
    if (S.pot != POT_SW) return;                 // uniform over the block
    const SWc<T> P = reinterpret_cast<const SWc<T>*>(b.swc)[S.prm];
    const int lane = threadIdx.x % L, grp = threadIdx.x / L;
    const int lbase = ((threadIdx.x & 31) / L) * L;
    const unsigned gmask = (L == 32) ? 0xffffffffu : (((1u << L) - 1u) << lbase);
    offset_table<T>(soff, pick<T>(st.h[0], st.h_f[0]), pick<T>(st.h[1], st.h_f[1]), pick<T>(st.h[2], st.h_f[2]));
    const int ia = part * G + grp;
    const bool valid = ia < ta.count;
    const int i = ta.first + ia;

    T fx = 0, fy = 0, fz = 0, en = 0;
    T w0 = 0, w1 = 0, w2 = 0, w3 = 0, w4 = 0, w5 = 0;
    if (valid) {
        const T4 xi = reinterpret_cast<const T4*>(b.xs)[i];
        const int ci = min(b.cnt[i], b.cap);
        T4* Fl = reinterpret_cast<T4*>(b.shd) + (size_t)i * kShell;
        int* Sj = b.shj + (size_t)i * kShell;
        // 1. compaction, NB row entries per lane in flight (row loads, then position gathers)
        constexpr int NB = (24 + L - 1) / L;
        int m = 0;
        for (int base = 0; base < ci; base += NB * L) {
            int e[NB];
            T4 xj[NB];
#pragma unroll
            for (int u = 0; u < NB; ++u) {
                const int sidx = base + u * L + lane;
                e[u] = sidx < ci ? b.nbr[nbr_at(b, i, sidx)] : 0;
                if (!NEFE_IN_RANGE(e[u] & (int)kIndexMask, b.ntot, &st.err)) e[u] = i;
            }
#pragma unroll
            for (int u = 0; u < NB; ++u)
                if (base + u * L + lane < ci) xj[u] = reinterpret_cast<const T4*>(b.xs)[e[u] & (int)kIndexMask];
#pragma unroll
            for (int u = 0; u < NB; ++u) {
                const int sidx = base + u * L + lane;
                bool in = false;
                T dx = 0, dy = 0, dz = 0, r2 = 0;
                if (sidx < ci) {
                    const T4 oh = soff[(unsigned)e[u] >> kCodeShift];
                    dx = (xj[u].x - xi.x) + oh.x;
                    dy = (xj[u].y - xi.y) + oh.y;
                    dz = (xj[u].z - xi.z) + oh.z;
                    r2 = dx * dx + dy * dy + dz * dz;
                    in = r2 < P.act2;
                }
                const unsigned bal = __ballot_sync(gmask, in);
                if (in) {
                    const int pos = m + __popc(bal & ((1u << (threadIdx.x & 31)) - 1u));
                    if (pos < kShell) {
                        sh_u[grp][pos] = mk4(dx, dy, dz, r2);
                        Sj[pos] = e[u] & (int)kIndexMask;
                    }
                }
                m += __popc(bal);
            }
        }
        if (m > kShell) {
            if (lane == 0) atomicOr(&st.err, NEFE_ERR_SHELL_OVERFLOW);
            m = kShell;
        }
        if (lane == 0 && m < kShell) Sj[m] = -1;
        __syncwarp(gmask);
        // 2. edges: pair terms, g, dg, unit vectors
        for (int a = lane; a < m; a += L) {
            const T4 d = sh_u[grp][a];
            const T ir = xrsqrt(d.w);
            const T r = d.w * ir;
            T phi, dphi, g, dg;
            sw_edge<T>(P, r, phi, dphi, g, dg);
            const T c = dphi * ir;
            fx += c * d.x; fy += c * d.y; fz += c * d.z;
            en += (T)0.5 * phi;
            const T hc = (T)-0.5 * c;
            w0 += hc * d.x * d.x; w1 += hc * d.y * d.y; w2 += hc * d.z * d.z;
            w3 += hc * d.x * d.y; w4 += hc * d.x * d.z; w5 += hc * d.y * d.z;
            sh_u[grp][a] = mk4(d.x * ir, d.y * ir, d.z * ir, r);
            sh_g[grp][a] = g;
            sh_dg[grp][a] = dg;
        }
        __syncwarp(gmask);
        // 3. leg forces
        for (int a = lane; a < m; a += L) {
            const T4 ua = sh_u[grp][a];
            const T ga = sh_g[grp][a];
            const T k1 = (T)2 * P.epslam * ga * xrcp(ua.w);
            const T k2 = P.epslam * sh_dg[grp][a];
            T ax = 0, ay = 0, az = 0, cc = 0, eh = 0;
            for (int bb = 0; bb < m; ++bb) {
                if (bb == a) continue;
                const T4 ub = sh_u[grp][bb];
                const T gb = sh_g[grp][bb];
                const T c = ua.x * ub.x + ua.y * ub.y + ua.z * ub.z;
                const T dc = c - P.c0;
                const T s1 = dc * gb;
                const T t1 = k1 * s1;
                ax += t1 * ub.x; ay += t1 * ub.y; az += t1 * ub.z;
                cc += t1 * c - k2 * dc * s1;
                const T hb = dc * s1;                    // (c - c0)^2 g_b
                eh += hb;
            }
            const T lx = cc * ua.x - ax, ly = cc * ua.y - ay, lz = cc * ua.z - az;
            Fl[a] = mk4(lx, ly, lz, (T)0);
            fx -= lx; fy -= ly; fz -= lz;
            const T hsum = (T)0.5 * P.epslam * ga * eh;  // half of every triplet (i; a, b), b != a
            en += hsum;
            const T dx = ua.x * ua.w, dy = ua.y * ua.w, dz = ua.z * ua.w;
            w0 += dx * lx; w1 += dy * ly; w2 += dz * lz;
            w3 += (T)0.5 * (dx * ly + dy * lx);
            w4 += (T)0.5 * (dx * lz + dz * lx);
            w5 += (T)0.5 * (dy * lz + dz * ly);
        }
        // the atom's force, energy and virial (summed over its lanes); pass B adds the energy
        // and virial to its block sums, so this pass has no block reduction
        T v[10] = {fx, fy, fz, en, w0, w1, w2, w3, w4, w5};
#pragma unroll
        for (int o = L / 2; o > 0; o >>= 1)
#pragma unroll
            for (int k = 0; k < 10; ++k) v[k] += __shfl_xor_sync(gmask, v[k], o);
        if (lane == 0) {
            T4* Pa = reinterpret_cast<T4*>(b.P);
            Pa[i] = mk4(v[0], v[1], v[2], v[3]);
            Pa[b.ntot + 2 * (size_t)i] = mk4(v[4], v[5], v[6], v[7]);
            Pa[b.ntot + 2 * (size_t)i + 1] = mk4(v[8], v[9], (T)0, (T)0);
            b.shn[i] = m;
        }
    }
}

// Force pass A, one thread per atom (64-thread blocks, half a tile each), FP32: the same
// three phases as k_edges with no lane coordination (no ballots, no idle lanes while another
// holds edges).  The shell is a column per thread: its first kShell1Shared entries in shared
// memory (20 bytes each; this table bounds the occupancy, so it is sized for the typical
// shell), the rest up to kShell1 in a per-atom spill area in global memory (b.spill; without
// one the capacity is kShell1Shared).  Loop counters are equal across a warp, so the choice
// between the two places is uniform.
constexpr int kShell1Shared = 8;
constexpr int kShell1 = kShell1Shared + kSpill1;
constexpr int kEdges1Threads = 64;

constexpr int kEdges1K1 = kShell1Shared;

// Pass A for atom i (thread-per-atom): compaction of its Verlet row into the in-cutoff shell
// (column t of the shared shell table, entries past its K1 rows in the global spill area), pair
// terms, and the leg forces of the triplets centred on i, stored per shell edge.
// pos(j) returns atom j's mirror position (from global memory or a shared copy).
template <typename T, int NT, typename PosFn>
__device__ __forceinline__ void edges1_atom(const Bufs& b, const SWc<T>& P, DevState& st,
                                            const T* soff, int i, int t,
                                            typename V4<T>::t (*sh_u)[NT], T (*sh_r)[NT], PosFn pos) {
    using T4 = typename V4<T>::t;
    constexpr int K1 = kShell1Shared, KS = kShell1 - kShell1Shared;
    const T4 xi = pos(i);
    const int ci = min(b.cnt[i], b.cap);
    const int* row = b.nbr + (size_t)i * b.cap;
    T4* Fl = reinterpret_cast<T4*>(b.shd) + (size_t)i * kShell;
    int* Sj = b.shj + (size_t)i * kShell;
    T4* spu = b.spill ? reinterpret_cast<T4*>(b.spill) + (size_t)i * KS : nullptr;
    T* spr = b.spill ? reinterpret_cast<T*>(reinterpret_cast<T4*>(b.spill) + (size_t)b.ntot * KS) + (size_t)i * KS
                     : nullptr;
    const int capm = b.spill ? kShell1 : K1;
    auto put_u = [&](int a, T4 v) { if (a < K1) sh_u[a][t] = v; else spu[a - K1] = v; };
    auto get_u = [&](int a) -> T4 { return a < K1 ? sh_u[a][t] : spu[a - K1]; };
    auto put_r = [&](int a, T v) { if (a < K1) sh_r[a][t] = v; else spr[a - K1] = v; };
    auto get_r = [&](int a) -> T { return a < K1 ? sh_r[a][t] : spr[a - K1]; };
    // 1. compaction, four row entries in flight.  Interleaved rows (engine): one 16-byte load
    // per four entries, contiguous across the warp, and the row is padded to a multiple of 4
    // with entries that fail the distance test, so every entry of the last group is read
    // unguarded.  Row-major rows: one 16-byte load when the row capacity is a multiple of 4,
    // entries past ci not used.
    int m = 0;
    const bool il = b.nbr_il != 0;
    const bool row4 = (b.cap & 3) == 0;
    const int cend = il ? (ci + 3) & ~3 : ci;
    const int4* row_il = reinterpret_cast<const int4*>(b.nbr) + i;
    for (int base = 0; base < cend; base += 4) {
        int e[4];
        T4 xj[4];
        if (il) {
            const int4 r4 = row_il[(size_t)(base >> 2) * b.ntot];
            e[0] = r4.x; e[1] = r4.y; e[2] = r4.z; e[3] = r4.w;
        } else if (row4) {
            const int4 r4 = *reinterpret_cast<const int4*>(row + base);
            e[0] = r4.x; e[1] = r4.y; e[2] = r4.z; e[3] = r4.w;
        } else {
#pragma unroll
            for (int u = 0; u < 4; ++u) e[u] = (base + u < ci) ? row[base + u] : 0;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (!NEFE_IN_RANGE(e[u] & (int)kIndexMask, b.ntot, &st.err)) e[u] = i;
#pragma unroll
        for (int u = 0; u < 4; ++u)
            if (il || base + u < ci) xj[u] = pos(e[u] & (int)kIndexMask);
#pragma unroll
        for (int u = 0; u < 4; ++u) {
            if (!il && base + u >= ci) continue;
            const unsigned c = (unsigned)e[u] >> kCodeShift;
            const T dx = (xj[u].x - xi.x) + soff[c], dy = (xj[u].y - xi.y) + soff[32 + c],
                    dz = (xj[u].z - xi.z) + soff[64 + c];
            const T r2 = dx * dx + dy * dy + dz * dz;
            if (r2 < P.act2) {
                if (m < capm) {
                    put_u(m, mk4(dx, dy, dz, r2));
                    Sj[m] = e[u] & (int)kIndexMask;
                }
                ++m;
            }
        }
    }
    if (m > capm) {
        atomicOr(&st.err, NEFE_ERR_SHELL_OVERFLOW);
        m = capm;
    }
    if (m < kShell) Sj[m] = -1;
    T fx = 0, fy = 0, fz = 0, en = 0;
    T w0 = 0, w1 = 0, w2 = 0, w3 = 0, w4 = 0, w5 = 0;
    // Moments of the shell: G = sum_b g_b, m1 = sum_b g_b u_b, M = sum_b g_b u_b u_b^T.  Every
    // sum over the partner edge b of a triplet (i; a, b) that the leg force needs is linear in
    // these, so the triplets of an atom cost O(m) instead of O(m^2) (see phase 3).
    T G = 0, m1x = 0, m1y = 0, m1z = 0, Mxx = 0, Myy = 0, Mzz = 0, Mxy = 0, Mxz = 0, Myz = 0;
    // 2. edges
    for (int a = 0; a < m; ++a) {
        const T4 d = get_u(a);
        const T ir = xrsqrt(d.w);
        const T r = d.w * ir;
        T phi, dphi, g, dg;
        sw_edge<T>(P, r, phi, dphi, g, dg);
        const T c = dphi * ir;
        fx += c * d.x; fy += c * d.y; fz += c * d.z;
        en += (T)0.5 * phi;
        const T hc = (T)-0.5 * c;
        w0 += hc * d.x * d.x; w1 += hc * d.y * d.y; w2 += hc * d.z * d.z;
        w3 += hc * d.x * d.y; w4 += hc * d.x * d.z; w5 += hc * d.y * d.z;
        const T ux = d.x * ir, uy = d.y * ir, uz = d.z * ir;
        put_u(a, mk4(ux, uy, uz, g));
        put_r(a, r);
        const T gx = g * ux, gy = g * uy, gz = g * uz;
        G += g; m1x += gx; m1y += gy; m1z += gz;
        Mxx += gx * ux; Myy += gy * uy; Mzz += gz * uz; Mxy += gx * uy; Mxz += gx * uz; Myz += gy * uz;
    }
    // 3. leg forces.  For edge a with c_b = u_a.u_b, over every partner b != a:
    //   S1 = sum g_b (c_b - c0) u_b = M u_a - c0 m1 - g_a (1 - c0) u_a,
    //   S2 = sum g_b (c_b - c0) c_b = u_a.M u_a - c0 u_a.m1 - g_a (1 - c0),
    //   S3 = sum g_b (c_b - c0)^2   = u_a.M u_a - 2 c0 u_a.m1 + c0^2 G - g_a (1 - c0)^2
    // (the sums over all b, minus the b = a term with c = 1).  The force the triplets (i; a, b)
    // exert on leg atom j_a is L_a = (k1 S2 - k2 S3) u_a - k1 S1 with k1 = 2 eps lambda g_a / r_a,
    // k2 = eps lambda dg_a/dr, and the atom's share of their energy is eps lambda g_a S3 / 2.
    const T c0 = P.c0, c02 = c0 * c0;
    for (int a = 0; a < m; ++a) {
        const T4 ua = get_u(a);
        const T ga = ua.w, ra = get_r(a);
        // dg/dr of edge a from g and r: -g gamma / (sigma (s - a)^2) (0 beyond the active cutoff)
        const T den = ra * P.inv_sig - P.a;
        const T ida = den < -cut_eps<T>() ? xrcp(den) : (T)0;
        const T dga = -ga * P.gam * ida * ida * P.inv_sig;
        const T k1 = (T)2 * P.epslam * ga * xrcp(ra);
        const T k2 = P.epslam * dga;
        const T Mux = Mxx * ua.x + Mxy * ua.y + Mxz * ua.z;
        const T Muy = Mxy * ua.x + Myy * ua.y + Myz * ua.z;
        const T Muz = Mxz * ua.x + Myz * ua.y + Mzz * ua.z;
        const T q = ua.x * Mux + ua.y * Muy + ua.z * Muz;
        const T pm = ua.x * m1x + ua.y * m1y + ua.z * m1z;
        const T self = ga * ((T)1 - c0);
        const T S2 = q - c0 * pm - self;
        const T S3 = q - (T)2 * c0 * pm + c02 * G - self * ((T)1 - c0);
        const T eh = S3;
        const T cc = k1 * S2 - k2 * S3;
        const T ax = k1 * (Mux - c0 * m1x - self * ua.x);
        const T ay = k1 * (Muy - c0 * m1y - self * ua.y);
        const T az = k1 * (Muz - c0 * m1z - self * ua.z);
        const T lx = cc * ua.x - ax, ly = cc * ua.y - ay, lz = cc * ua.z - az;
        Fl[a] = mk4(lx, ly, lz, (T)0);
        fx -= lx; fy -= ly; fz -= lz;
        en += (T)0.5 * P.epslam * ga * eh;
        const T dx = ua.x * ra, dy = ua.y * ra, dz = ua.z * ra;
        w0 += dx * lx; w1 += dy * ly; w2 += dz * lz;
        w3 += (T)0.5 * (dx * ly + dy * lx);
        w4 += (T)0.5 * (dx * lz + dz * lx);
        w5 += (T)0.5 * (dy * lz + dz * ly);
    }
    T4* Pa = reinterpret_cast<T4*>(b.P);
    Pa[i] = mk4(fx, fy, fz, en);
    Pa[b.ntot + 2 * (size_t)i] = mk4(w0, w1, w2, w3);
    Pa[b.ntot + 2 * (size_t)i + 1] = mk4(w4, w5, (T)0, (T)0);
    b.shn[i] = m;
}

template <typename T>
__global__ void __launch_bounds__(kEdges1Threads, 16) k_edges1(Bufs b) {
    dep_wait();
    using T4 = typename V4<T>::t;
    constexpr int NT = kEdges1Threads, IPT = kTile / NT;
    __shared__ T4 sh_u[kEdges1K1][NT];           // (d, r^2) after compaction, then (u, g)
    __shared__ T sh_r[kEdges1K1][NT];            // r
    __shared__ T soff[3 * 32];
    const TileAtom ta = tile_of(b, (int)blockIdx.x / IPT + b.tile_base);
    const DevSys& S = b.sys[ta.sys];
    DevState& st = b.st[ta.sys];
    if (S.pot != POT_SW) return;                 // uniform over the block
    const SWc<T> P = reinterpret_cast<const SWc<T>*>(b.swc)[S.prm];
    offset_rows<T>(soff, pick<T>(st.h[0], st.h_f[0]), pick<T>(st.h[1], st.h_f[1]), pick<T>(st.h[2], st.h_f[2]));
    const int t = threadIdx.x;
    const int ia = ((int)blockIdx.x % IPT) * NT + t;
    if (ia < ta.count) {
        const T4* X = reinterpret_cast<const T4*>(b.xs);
        edges1_atom<T, NT>(b, P, st, soff, ta.first + ia, t, sh_u, sh_r, [X](int j) { return X[j]; });
    }
}

// ------------------------------------------------------------------------------------
// Scatter form of the force passes (FP32): pass A adds the force that each atom's terms exert on
// each leg atom, and minus their sum on the atom itself, into per-atom int32 accumulators (units of
// 2^-22 eV/A for silicon) with global reductions.  Integer addition is associative, so the result does not
// depend on the order in which the reductions arrive (bitwise reproducible), and no second pass has
// to find the legs again: a streaming epilogue (k_finish) reads and clears each accumulator.
// The x and y terms travel in one 64-bit reduction as y 2^32 + x (two's complement, modulo
// 2^64): integer addition is linear, so the 64-bit word accumulates Y 2^32 + X exactly, X and Y
// being the int32 sums.  Its low word is X; its high word is Y - 1 when X < 0 (the borrow), which
// the reader undoes (force_of_acc).  Two reductions per force instead of three.
// The unit follows the potential: 2^-22 eV/A times a power of two near (eps/sigma) / (silicon's), see
// leg_power, so that the rounding is relative to the potential's own forces (with eps a hundredth of
// silicon's a fixed unit left 2e-5 of the largest force).  In these units:
// a term of kLegFine eV/A or more is split: its multiples of kLegCoarse go to a second accumulator
// (int64, one count per multiple) and the rest, at most 7.5 eV/A, stays; up to 64 rests (32 legs, 32 own
// edges) fit the int32 sum.  The second accumulator is read only for tiles whose flag says that
// something was added (at 1000 K some atom of a system of thousands has such a term on most steps,
// but few tiles do).  A term that is not finite, or of kLegMax (2.5e17 eV/A) and more, sets the atom's
// count to kLegNan, from which no sum of counts (64 terms of up to 2^54) comes back below kLegLost:
// the force is NaN, as a floating-point sum would have it.
// ------------------------------------------------------------------------------------
constexpr float kLegCoarse = 14.0f;
constexpr float kLegMax = 14.0f * 18014398509481984.0f;   // 14 2^54
constexpr long long kLegNan = 1LL << 62, kLegLost = 1LL << 61;
constexpr float kLegRefuse = 48.0f;
constexpr float kPairOdd = 6.0f;                 // half a pair force above which an own sum could reach kLegRefuse

// Splits a large term into n multiples of kLegCoarse and the rest (n = kLegNan: out of range or not
// finite).  A count above 2^24 is rounded; what it leaves is split again.  Each remainder is an FP32
// number, and the last is at most 7.5.
__device__ __forceinline__ float split_term(float v, long long& n) {
    n = 0;
    if (!(fabsf(v) < kLegMax)) {
        n = kLegNan;
        return 0.0f;
    }
    while (fabsf(v) > 7.5f) {
        const float h = rintf(v * (1.0f / kLegCoarse));
        v = fmaf(-kLegCoarse, h, v);
        n += fabsf(h) < 1e9f ? (long long)(int)h : (long long)h;
    }
    return v;
}

// n multiples of kLegCoarse for component k of atom j.
__device__ __forceinline__ void add_count(const Bufs& b, const DevSys& S, int j, int k, long long n) {
    unsigned long long* hi = reinterpret_cast<unsigned long long*>(b.lacc_hi + 3 * (size_t)j) + k;
    if (n == kLegNan || n == -kLegNan) atomicExch(hi, (unsigned long long)kLegNan);
    else atomicAdd(hi, (unsigned long long)n);
    b.hi_flag[S.tile0 + (j - S.off) / kTile] = 1;
}

__device__ __forceinline__ void red_force(int* acc4, int x, int y, int z) {
    const unsigned long long xy = ((unsigned long long)(long long)y << 32) + (unsigned long long)(long long)x;
    atomicAdd(reinterpret_cast<unsigned long long*>(acc4), xy);
    atomicAdd(acc4 + 2, z);
}

// The int32 sums (X, Y, Z) of an accumulator written by red_force.
__device__ __forceinline__ int3 force_of_acc(int4 q) {
    return make_int3(q.x, q.y + (q.x < 0 ? 1 : 0), q.z);
}

// Force pass A, scatter form.  Each warp takes G = 32, 16 or 8 consecutive atoms, 32 / G lanes to an
// atom.
//   1. The lanes walk the atoms' Verlet rows and mark the entries inside the cutoff.  Positions are
//      fractions: the difference of two is the nearest image by itself, so no cell offsets are looked
//      up.  This filter reads 8-byte positions (21 bits an axis) and keeps a margin for their rounding.
//   2. The marked entries become one edge list of the warp, taken 32 at a time: unit vector and g from
//      the full positions (resolution L 2^-32); an edge of the margin has no terms.
//   3. Per atom: the shell's moments.
//   4. The edge list again: pair terms and leg forces (see sw_leg), quantised and added to the leg
//      atoms; the own sums through shared integer accumulators.
// What bounds it is the L1 wavefronts of the position gathers (17 a warp for 16-byte positions of 32
// scattered atoms; step 1 alone took 83 of 172 us with them), hence the 8-byte ones.  With one thread
// per atom throughout (the form before), steps 2 and 4 ran at the largest shell of each warp (9 edges
// for a mean of 5.8) with idle lanes, and shells above 8 edges spilled to global memory.  Appending to
// the list during the walk instead of marking (no second read of rows and positions) was slower by 10 us.
// G: 32 where that gives every SM kScatterFull warps; smaller systems take 16 or 8 atoms to a warp,
// whose chain of row groups and edge iterations is shorter by as much (8000 atoms: 8.9 -> 6.8 us).
// A list holds kListEdges edges; atoms whose edges do not fit wait for the next batch.
// Against the forms before, live in the step: 1,024,000-atom crystal at skin 1.6 A (28 row entries, 5.8
// edges an atom) 171.5 -> 151 us, or 167 with leg_refuse (its screen has the own sums of a warp computed
// again wherever half a pair force reaches 6 eV/A); 1,008,516 atoms of diamond / beta-tin pairs (12.8
// edges), with leg_refuse, 308-357 -> 232-255 us; against the gather form's two passes, 96,000 atoms under
// barostats 85 -> 50 us, 8000 atoms 22.9 -> 19.4.
constexpr int kListEdges = 224;         // 32 atoms of a crystal hold 186 +- 5; smaller lists leave more L1 and warps
constexpr int kEdgesDBlocks = 7;         // blocks of k_edges_d an SM holds (shared memory)
// The atoms of a block of the edge-list kernels: of tile `tile`, from atom `first` on, 2^lg to a warp.
// Tiles from b.tail_tile on are cut finer (2^lg_tail): see set_edge_items.
struct EdgeItem {
    int lg, tile, first;
};
__device__ __forceinline__ EdgeItem edge_item(const Bufs& b) {
    const int big = max(0, b.tail_tile - b.tile_base), nbig = big << (6 - b.lg);
    const bool tail = (int)blockIdx.x >= nbig;
    const int lg = tail ? b.lg_tail : b.lg, item = (int)blockIdx.x - (tail ? nbig : 0);
    return {lg, b.tile_base + (tail ? big : 0) + (item >> (6 - lg)), (item & ((64 >> lg) - 1)) << (lg + 1)};
}
constexpr int kScatterThreads = 64;
// Resident blocks per SM the registers are bounded for: 14 where the launch fills them (crystal 154.7
// us, 12: 159.6), else as many registers as the kernel wants (12 blocks' worth: 6.8 against 7.4 us for
// 8000 atoms).
constexpr int kScatterBlocks = 14, kScatterBlocksFew = 10;
template <bool EATOM>
struct __align__(16) ScatterShared {
    float4 u[kListEdges];            // unit vector, g
    float r[kListEdges];
    unsigned id[kListEdges];         // atom of the warp << 27 | leg atom
    float4 mom[3][32];               // moments; before them, the atoms' positions
    int own[3][32];
    float e[EATOM ? kListEdges : 1];
};

// r/sigma - a, from constants of twice the precision.
__device__ __forceinline__ float below_cut(const SWc<float>& P, float r) {
    return fmaf(r, P.inv_sig, -P.a) + fmaf(r, P.inv_sig_lo, -P.a_lo);
}

// Pair term of an edge (r < s_act sigma) and what the leg force needs of g: phi, dphi/dr, 1/(s - a).
__device__ __forceinline__ void pair_edge(const SWc<float>& P, float r, float& phi, float& dphi, float& id) {
    const float s = r * P.inv_sig, den = below_cut(P, r);
    const bool in = s < P.s_act && den < -cut_eps<float>();
    id = in ? xrcp(den) : 0.0f;
    float e1 = in ? xexp(id) : 0.0f;
    float rp, rq;
    const float is = xrcp(s);
    if (P.int_pq) {
        const float is2 = xrcp(s * s);
        rp = is2 * is2;
        rq = 1.0f;
    } else {
        rp = xpow(s, -P.p);
        rq = xpow(s, -P.q);
    }
    const float poly = fmaf(P.B, rp, -rq) + P.B_lo * rp;
    e1 *= P.epsA;
    phi = poly * e1;
    dphi = e1 * ((P.q * rq - P.p * fmaf(P.B, rp, P.B_lo * rp)) * is - poly * id * id) * P.inv_sig;
}

// An edge's terms in the last phase: the force on the leg atom (see sw_leg; the rows of the shell's
// moments M, m1 are ma, mb, mc), half the pair force, energies and 1/(s - a).
struct LegOut {
    float x, y, z, hp, phi, s3, ida;
};
__device__ __forceinline__ LegOut leg_of_edge(const SWc<float>& P, const float4& ua, float ra, const float4& ma,
                                              const float4& mb, const float4& mc, float G) {
    LegOut o;
    float dphi;
    pair_edge(P, ra, o.phi, dphi, o.ida);
    o.hp = 0.5f * dphi;
    const float c0 = P.c0, ga = ua.w;
    const float eg = P.epslam * ga;
    const float k1 = 2.0f * eg * xrcp(ra);
    const float k2 = -eg * P.gam * o.ida * o.ida * P.inv_sig;
    const float Mux = ma.x * ua.x + ma.y * ua.y + ma.z * ua.z;
    const float Muy = mb.x * ua.x + mb.y * ua.y + mb.z * ua.z;
    const float Muz = mc.x * ua.x + mc.y * ua.y + mc.z * ua.z;
    const float q = ua.x * Mux + ua.y * Muy + ua.z * Muz;
    const float pm = ua.x * ma.w + ua.y * mb.w + ua.z * mc.w;
    const float self = ga * (1.0f - c0);
    const float S2 = q - c0 * pm - self;
    o.s3 = q - 2.0f * c0 * pm + c0 * c0 * G - self * (1.0f - c0);
    const float cc = k1 * S2 - k2 * o.s3 - o.hp;
    o.x = cc * ua.x - k1 * (Mux - c0 * ma.w - self * ua.x);
    o.y = cc * ua.y - k1 * (Muy - c0 * mb.w - self * ua.y);
    o.z = cc * ua.z - k1 * (Muz - c0 * mc.w - self * ua.z);
    return o;
}

// Rare: the edges whose terms have to be split (or, with leg_refuse, whose triplet part may be refused): bit k
// of `odd` is edge 32 k + lane of the warp's list.  This comes after the edge loop, which leaves the force in
// sh.u (leg_refuse: it is computed again): a call in the middle of the loop had the compiler spill (16 to 68
// bytes by what was called; 64 pairs 64.9 ms a pass with 16, 67.1 with 68, 63.7 with none).  All lanes
// of the warp come here; i0: the warp's first atom, Gm: the lane's atom's moment.
template <bool EATOM>
__device__ __forceinline__ void add_large_legs(const Bufs& b, const DevSys& S, const SWc<float>& P, ScatterShared<EATOM>& sh,
                                            int lane, int i0, unsigned odd, float Gm, unsigned* err) {
    const float unit = P.leg_scale / kLegScale;
    for (unsigned any = __reduce_or_sync(0xffffffffu, odd); any; any &= any - 1u) {
        const int q = __ffs(any) - 1, e = 32 * q + lane;
        const bool on = (odd >> q & 1u) != 0u;
        const unsigned w = on ? sh.id[e] : 0u;
        const int t = (int)(w >> kCodeShift), j = (int)(w & kIndexMask), i = i0 + t;
        const float Gt = __shfl_sync(0xffffffffu, Gm, t);
        if (!on) continue;
        const float4 u = sh.u[e];
        float l[3] = {u.x, u.y, u.z}, p[3];      // p: what the leg atom gets
        bool same = true;
        if (b.leg_refuse) {
            const LegOut o = leg_of_edge(P, u, sh.r[e], sh.mom[0][t], sh.mom[1][t], sh.mom[2][t], Gt);
            l[0] = o.x; l[1] = o.y; l[2] = o.z;
            same = fabsf(o.x + o.hp * u.x) < kLegRefuse && fabsf(o.y + o.hp * u.y) < kLegRefuse &&
                   fabsf(o.z + o.hp * u.z) < kLegRefuse;
            p[0] = -o.hp * u.x; p[1] = -o.hp * u.y; p[2] = -o.hp * u.z;
            if (!same) atomicOr(err, NEFE_ERR_NAN);
        }
        int ql[3], qp[3];
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            long long nl, np;
            ql[k] = qp[k] = __float2int_rn(split_term(l[k] * unit, nl) * kLegScale);
            np = nl;
            if (!same) qp[k] = __float2int_rn(split_term(p[k] * unit, np) * kLegScale);
            if (nl == kLegNan || np == kLegNan) {
                atomicOr(err, NEFE_ERR_NAN);
                if (b.leg_refuse) {              // (a refused term is left out)
                    nl = nl == kLegNan ? 0 : nl;
                    np = np == kLegNan ? 0 : np;
                }
            }
            if (np) add_count(b, S, j, k, np);
            if (nl) add_count(b, S, i, k, -nl);
            atomicAdd(&sh.own[k][t], ql[k]);
        }
        red_force(b.lacc + 4 * (size_t)j, qp[0], qp[1], qp[2]);
    }
    __syncwarp();
}

// Rare: takes the own sum of an atom (its pair forces and the recoils of its triplet legs, sum of
// hp u - l) out again if it is refused.  All lanes of the warp call it; part, t: the lane's part and
// atom, m: its edges (on: in this batch), G: atoms.
template <bool EATOM>
__device__ __noinline__ void refuse_own(const Bufs& b, const DevSys& S, const SWc<float>& P, ScatterShared<EATOM>& sh,
                                        int lane, int G, int i, int m, int mx, float Gm, unsigned* err) {
    const int t = lane & (G - 1);
    float ox = 0.0f, oy = 0.0f, oz = 0.0f;
    int base = 0;
    for (int a = 0; a < mx; ++a) {
        const unsigned bal = __ballot_sync(0xffffffffu, a < m);
        if (a < m) {
            const int e = base + __popc(bal & ((1u << lane) - 1u));
            const float4 u = sh.u[e];
            const LegOut o = leg_of_edge(P, u, sh.r[e], sh.mom[0][t], sh.mom[1][t], sh.mom[2][t], Gm);
            ox += o.hp * u.x - o.x; oy += o.hp * u.y - o.y; oz += o.hp * u.z - o.z;
        }
        base += __popc(bal);
    }
    for (int o = 16; o >= G; o >>= 1) {
        ox += __shfl_xor_sync(0xffffffffu, ox, o);
        oy += __shfl_xor_sync(0xffffffffu, oy, o);
        oz += __shfl_xor_sync(0xffffffffu, oz, o);
    }
    if (lane < G && !(fabsf(ox) < kLegRefuse && fabsf(oy) < kLegRefuse && fabsf(oz) < kLegRefuse)) {
        atomicOr(err, NEFE_ERR_NAN);
        const float unit = P.leg_scale / kLegScale, o[3] = {ox * unit, oy * unit, oz * unit};
        for (int k = 0; k < 3; ++k) {
            long long n;
            sh.own[k][t] += __float2int_rn(split_term(o[k], n) * kLegScale);
            if (n && n != kLegNan) add_count(b, S, i, k, -n);
        }
    }
    __syncwarp();
}

// Step 1 of the edge-list kernels for atom i: the lane takes the row's octets part, part + 2^lpa, ...
// and marks their entries closer than sqrt(rc2) (with the margin of the packed positions): entry
// 8 (part + n 2^lpa) + k is bit 8 n + k of (lo, hi).
__device__ __forceinline__ void mark_row(const Bufs& b, int i, int part, int lpa, const float4& L, float rc2, unsigned* err,
                                         unsigned& lo, unsigned& hi) {
    const bool il = b.nbr_il != 0, wide = il || b.row4;
    const int4* rows4 = il ? reinterpret_cast<const int4*>(b.nbr) + i : reinterpret_cast<const int4*>(b.nbr + (size_t)i * b.cap);
    const size_t rstep = il ? (size_t)b.ntot : 1;
    const uint2* X = b.xc;
    const uint2 pi = X[i];
    const int xi = (int)pi.y, yi = (int)__funnelshift_l(pi.x, pi.y, 21), zi = (int)(pi.x << 10);
    const int ci = min(b.cnt[i], b.cap);
    // each axis of the packed difference is within 2 units of 2^-21 L of the true one
    const float mg = 2.0f * 2048.0f * (L.x + L.y + L.z);
    const float rc = sqrtf(rc2) + mg, act2 = rc * rc;
    int shift = 0;
    for (int base = 8 * part; base < ci; base += 8 << lpa, shift += 8) {
        int e[8];
#pragma unroll
        for (int v = 0; v < 8; v += 4) {
            if (wide) {
                int4 r = make_int4(i, i, i, i);
                if (base + v < ci) r = rows4[(size_t)((base + v) >> 2) * rstep];
                e[v] = r.x; e[v + 1] = r.y; e[v + 2] = r.z; e[v + 3] = r.w;
            } else {
                const int* row = reinterpret_cast<const int*>(rows4);
#pragma unroll
                for (int u = v; u < v + 4; ++u) e[u] = base + u < ci ? row[base + u] : i;
            }
        }
        unsigned oct = 0u;
        uint2 pj[8];
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            // past the row's length a row-major group holds the caller's bytes: not an index
            int j = (il || base + u < ci) ? (e[u] & (int)kIndexMask) : i;
            if (!NEFE_IN_RANGE(j, b.ntot, err)) j = i;
            pj[u] = X[j];
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
            const float dx = (float)wrap_sub((int)pj[u].y, xi) * L.x,
                        dy = (float)wrap_sub((int)__funnelshift_l(pj[u].x, pj[u].y, 21), yi) * L.y,
                        dz = (float)wrap_sub((int)(pj[u].x << 10), zi) * L.z;
            if (dx * dx + dy * dy + dz * dz < act2) oct |= 1u << u;
        }
        // entries past the length are the atom itself
        if (ci - base < 8) oct &= (1u << (ci - base)) - 1u;
        if (shift < 32) lo |= oct << shift; else hi |= oct << (shift - 32);
    }
}

// COMMON: every system has the same potential constants, which are then kernel arguments (operands of
// the constant bank, no loads: 171 -> 155 us on the crystal); otherwise they are read from the table.
// FINE: positions carry ten more bits an axis (a test in the loop cost 8000 atoms 1.4 %).
template <bool EATOM, bool GRAD, bool COMMON, int BLOCKS, bool FINE>
__global__ void __launch_bounds__(kScatterThreads, BLOCKS)
k_edges_s(const __grid_constant__ Bufs b, const __grid_constant__ SWc<float> Pc) {
    dep_wait();
    constexpr unsigned kAll = 0xffffffffu;
    const EdgeItem it = edge_item(b);
    const int lg = it.lg, G = 1 << lg, lpa = 5 - lg;
    __shared__ ScatterShared<EATOM> shm[kScatterThreads / 32];
    ScatterShared<EATOM>& sh = shm[threadIdx.x >> 5];
    static_assert(kScatterThreads == 64 && kTile == 128, "two warps of 2^lg atoms a block");
    const TileAtom ta = tile_of(b, it.tile);
    const DevSys& S = b.sys[ta.sys];
    DevState& st = b.st[ta.sys];
    if (S.pot != POT_SW) return;                 // uniform over the block
    const SWc<float>& P = COMMON ? Pc : reinterpret_cast<const SWc<float>*>(b.swc)[S.prm];
    const int lane = threadIdx.x & 31, t = lane & (G - 1);
    const unsigned below = (1u << lane) - 1u;
    const int ia = it.first + ((int)(threadIdx.x >> 5) << lg) + t;   // of the tile
    const int i = ta.first + ia;
    const bool valid = ia < ta.count;
    // L 2^-32 to twice the precision: a relative error of L alone would be a uniform strain of up to
    // 6e-8, which the pressure sees (the row filter does without the second part)
    const float4 Lh = b.lscale[4 * ta.sys], Ll = b.lscale[4 * ta.sys + 1];
    // 1. accepted row entries
    unsigned lo = 0u, hi = 0u;
    if (valid) mark_row(b, i, lane >> lg, lpa, Lh, P.act2, &st.err, lo, hi);
    const int ml = __popc(lo) + __popc(hi);      // edges of this lane, then of its atom
    int m = ml;
    for (int o = 16; o >= G; o >>= 1) m += __shfl_xor_sync(kAll, m, o);
    int incl = m;                                // edges of atoms 0 .. t
    for (int o = 1; o < G; o <<= 1) {
        const int y = __shfl_up_sync(kAll, incl, o, G);
        if (t >= o) incl += y;
    }
    const int total = __shfl_sync(kAll, incl, G - 1);
    float red8[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};   // energy, -, virial
    float gth[7] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
    float en = 0.0f;
    int mtrue = 0;                               // edges of the lane inside the cutoff
    const float pair_odd = b.leg_refuse ? kPairOdd : INFINITY;
    const float fine = b.leg_refuse ? fminf(P.leg_fine, kLegFine) : P.leg_fine;   // (a refusal is in eV/A)
    int4* spos = reinterpret_cast<int4*>(&sh.mom[0][0]);
    sh.own[0][lane] = 0; sh.own[1][lane] = 0; sh.own[2][lane] = 0;
    for (int done = 0; done < total;) {
        const bool act = incl - m >= done && incl - done <= kListEdges && m > 0;
        const int ma = act ? ml : 0;
        const int mx = __reduce_max_sync(kAll, ma);
        int E = 0;
        {
            const int part = lane >> lg;
            unsigned l = lo, h = hi;
            for (int a = 0; a < mx; ++a) {       // slot by slot: consecutive lanes hold distinct atoms
                const bool on = a < ma;
                const unsigned bal = __ballot_sync(kAll, on);
                if (on) {
                    int k;
                    if (l) { k = __ffs(l) - 1; l &= l - 1u; }
                    else { k = 31 + __ffs(h); h &= h - 1u; }
                    k = 8 * (((k >> 3) << lpa) + part) + (k & 7);
                    int j = b.nbr[nbr_at(b, i, k)] & (int)kIndexMask;
                    if (!NEFE_IN_RANGE(j, b.ntot, &st.err)) j = i;
                    sh.id[E + __popc(bal & below)] = (unsigned)t << kCodeShift | (unsigned)j;
                }
                E += __popc(bal);
            }
        }
        if (lane < G && valid) spos[lane] = b.xf[i];
        __syncwarp();
        // 2. unit vectors and g; two edges a lane, so that their gathers are in flight together
        for (int e0 = lane; e0 < E; e0 += 64) {
            int4 xj[2], xi[2];
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const unsigned w = sh.id[e0 + 32 * u < E ? e0 + 32 * u : e0];
                xj[u] = b.xf[w & kIndexMask];
                xi[u] = spos[w >> kCodeShift];
            }
#pragma unroll
            for (int u = 0; u < 2; ++u) {
                const int e = e0 + 32 * u;
                if (e >= E) break;
                float fx = (float)wrap_sub(xj[u].x, xi[u].x), fy = (float)wrap_sub(xj[u].y, xi[u].y),
                      fz = (float)wrap_sub(xj[u].z, xi[u].z);
                if constexpr (FINE) {
                    const float3 g = frac_low_diff(xj[u].w, xi[u].w);
                    fx += g.x; fy += g.y; fz += g.z;
                }
                const float dx = fx * Lh.x + fx * Ll.x, dy = fy * Lh.y + fy * Ll.y, dz = fz * Lh.z + fz * Ll.z;
                const float r2 = dx * dx + dy * dy + dz * dz;
                // one Newton step: the hardware value's bias of a fraction of 1e-7 would scale every
                // edge alike, which the pressure sees
                float ir = xrsqrt(r2);
                ir = fmaf(0.5f * ir, fmaf(-r2 * ir, ir, 1.0f), ir);
                const float r = r2 * ir, s = r * P.inv_sig, den = below_cut(P, r);
                const float g = s < P.s_act && den < -cut_eps<float>() ? xexp(P.gam * xrcp(den)) : 0.0f;
                sh.u[e] = make_float4(dx * ir, dy * ir, dz * ir, g);
                sh.r[e] = r;
            }
        }
        __syncwarp();
        // 3. moments
        float Gm = 0;
        {
            float mx_ = 0, my = 0, mz = 0, xx = 0, yy = 0, zz = 0, xy = 0, xz = 0, yz = 0;
            int base = 0;
            for (int a = 0; a < mx; ++a) {
                const bool on = a < ma;
                const unsigned bal = __ballot_sync(kAll, on);
                if (on) {
                    const float4 u = sh.u[base + __popc(bal & below)];
                    const float gx = u.w * u.x, gy = u.w * u.y, gz = u.w * u.z;
                    mtrue += u.w > 0.0f ? 1 : 0;
                    Gm += u.w; mx_ += gx; my += gy; mz += gz;
                    xx += gx * u.x; yy += gy * u.y; zz += gz * u.z; xy += gx * u.y; xz += gx * u.z; yz += gy * u.z;
                }
                base += __popc(bal);
            }
            for (int o = 16; o >= G; o >>= 1) {
                Gm += __shfl_xor_sync(kAll, Gm, o);
                mx_ += __shfl_xor_sync(kAll, mx_, o); my += __shfl_xor_sync(kAll, my, o); mz += __shfl_xor_sync(kAll, mz, o);
                xx += __shfl_xor_sync(kAll, xx, o); yy += __shfl_xor_sync(kAll, yy, o); zz += __shfl_xor_sync(kAll, zz, o);
                xy += __shfl_xor_sync(kAll, xy, o); xz += __shfl_xor_sync(kAll, xz, o); yz += __shfl_xor_sync(kAll, yz, o);
            }
            if (lane < G) {
                sh.mom[0][t] = make_float4(xx, xy, xz, mx_);
                sh.mom[1][t] = make_float4(xy, yy, yz, my);
                sh.mom[2][t] = make_float4(xz, yz, zz, mz);
            }
        }
        __syncwarp();
        // 4. pair terms and leg forces
        unsigned odd = 0u;                       // edges whose terms are large (bit e / 32)
        static_assert(kListEdges <= 32 * 32, "a bit for each turn");
        for (int e0 = 0; e0 < E; e0 += 32) {
            const int e = e0 + lane;
            const bool on = e < E;
            const unsigned w = on ? sh.id[e] : 0u;
            const int te = (int)(w >> kCodeShift);
            const float Gt = __shfl_sync(kAll, Gm, te);
            if (!on) continue;
            const int j = (int)(w & kIndexMask);
            const float4 ua = sh.u[e];
            const float ra = sh.r[e];
            const LegOut o = leg_of_edge(P, ua, ra, sh.mom[0][te], sh.mom[1][te], sh.mom[2][te], Gt);
            const float h = P.epslam * ua.w * o.s3;   // the triplets of edge a, each seen from both its edges
            const float ee = 0.5f * (o.phi + h);
            red8[0] += ee;
            if (EATOM) sh.e[e] = ee;
            const float dx = ua.x * ra, dy = ua.y * ra, dz = ua.z * ra;
            red8[2] += dx * o.x; red8[3] += dy * o.y; red8[4] += dz * o.z;
            red8[5] += 0.5f * (dx * o.y + dy * o.x);
            red8[6] += 0.5f * (dx * o.z + dz * o.x);
            red8[7] += 0.5f * (dy * o.z + dz * o.y);
            if constexpr (GRAD) {
                float pg[5];
                sw_pair_pgrad<float>(P, ra, pg);
#pragma unroll
                for (int q5 = 0; q5 < 5; ++q5) gth[q5] += 0.5f * pg[q5];
                gth[4] += h * P.gam * o.ida * o.ida;
                gth[5] += 0.5f * P.eps * ua.w * o.s3;
                gth[6] += h * o.ida;
            }
            if (!(fabsf(o.x) < fine && fabsf(o.y) < fine && fabsf(o.z) < fine && fabsf(o.hp) < pair_odd)) {
                odd |= 1u << (e0 >> 5);
                if (!b.leg_refuse) sh.u[e] = make_float4(o.x, o.y, o.z, 0.0f);
                continue;
            }
            const int qx = __float2int_rn(o.x * P.leg_scale), qy = __float2int_rn(o.y * P.leg_scale),
                      qz = __float2int_rn(o.z * P.leg_scale);
            red_force(b.lacc + 4 * (size_t)j, qx, qy, qz);
            atomicAdd(&sh.own[0][te], qx);
            atomicAdd(&sh.own[1][te], qy);
            atomicAdd(&sh.own[2][te], qz);
        }
        __syncwarp();
        if (__any_sync(kAll, odd != 0u)) {
            add_large_legs(b, S, P, sh, lane, i - t, odd, Gm, &st.err);
            if (b.leg_refuse) refuse_own(b, S, P, sh, lane, G, i, ma, mx, Gm, &st.err);
        }
        if (EATOM) {                             // per-atom energies in slot order
            int base = 0;
            for (int a = 0; a < mx; ++a) {
                const unsigned bal = __ballot_sync(kAll, a < ma);
                if (a < ma) en += sh.e[base + __popc(bal & below)];
                base += __popc(bal);
            }
        }
        done = __reduce_max_sync(kAll, act ? incl : 0);
        __syncwarp();
    }
    __syncwarp();
    for (int o = 16; o >= G; o >>= 1) {
        mtrue += __shfl_xor_sync(kAll, mtrue, o);
        if (EATOM) en += __shfl_xor_sync(kAll, en, o);
    }
    if (lane < G && valid) {
        b.shn[i] = mtrue;
        if (mtrue > kShell) atomicOr(&st.err, NEFE_ERR_SHELL_OVERFLOW);
        if (m > 0) red_force(b.lacc + 4 * (size_t)i, -sh.own[0][lane], -sh.own[1][lane], -sh.own[2][lane]);
        if (EATOM && b.e_atom) b.e_atom[i] = (double)en;
    }
    long long* acc = b.acc + (size_t)ta.sys * ACC_N * kSlots;
    block_sum_to_acc<float, 8>(red8, acc, ACC_UINT, &st.err);
    if constexpr (GRAD) block_sum_to_acc<float, 7>(gth, acc, ACC_DTH, &st.err);
}

// Force pass A in FP64: the same edge list, with the terms of nefe_sw_terms.h.  The row filter is FP32, so
// FP64 (2 lanes a cycle and SM) sees only the edges; they are walked 32 at a time, and the triplets of
// an atom cost O(m).  Leg forces (each with half of its pair force) are stored per shell slot for pass
// B, the atom's own force is minus their sum; energy and virial go to the system's sums here.
// What bounds it is FP64 issue: about 160 operations an edge.  The form before computed distances of
// all row entries, divided and took the exponentials on partly idle lanes, and every triplet pair:
// 16 x 8000 atoms 988 -> 384 us, with dE/dtheta 32,768 liquid atoms 736 -> 268 us.
constexpr int kListEdgesD = 192;
struct __align__(16) EdgesDShared {
    double v[8][kListEdgesD];        // unit vector, 1/r, 1/(s - a), g, dphi, r; then the leg force
    unsigned id[kListEdgesD];        // atom of the warp << 27 | leg atom
    unsigned short slot[kListEdgesD];   // cell-offset code << 8 | shell slot
    double mom[10][32];
};
// Takes the marked entries at or beyond the cutoff (in the filter's margin) out of (lo, hi).  Only where
// an atom has more marked entries than its shell holds: a shell's slots are for edges.
__device__ __noinline__ void drop_margin(const Bufs& b, const DevState& st, double rc2, int i, int part, int lpa, unsigned& lo,
                                         unsigned& hi) {
    const double4* X = reinterpret_cast<const double4*>(b.xs);
    const double4 xi = X[i];
    unsigned w[2] = {lo, hi};
    for (int q = 0; q < 2; ++q)
        for (unsigned left = w[q]; left; left &= left - 1u) {
            const int bit = __ffs(left) - 1, k = bit + 32 * q;
            const unsigned e = (unsigned)b.nbr[nbr_at(b, i, 8 * (((k >> 3) << lpa) + part) + (k & 7))];
            int j = (int)(e & kIndexMask);
            if (j >= b.ntot) j = i;
            const int code = (int)(e >> kCodeShift);
            const double4 xj = X[j];
            const double dx = (xj.x - xi.x) + (code % 3 - 1) * st.h[0], dy = (xj.y - xi.y) + ((code / 3) % 3 - 1) * st.h[1],
                         dz = (xj.z - xi.z) + (code / 9 - 1) * st.h[2];
            if (dx * dx + dy * dy + dz * dz >= rc2) w[q] &= ~(1u << bit);
        }
    lo = w[0];
    hi = w[1];
}
// The next step's thermostat noise of 32 atoms (a quarter of a tile, one warp per Box-Muller pair) into
// xi_next, by blocks of pass A beyond the edges' own.  It depends on the step and the atom only, and in
// a small context it is the longest part of k_kick_drift (a chain of FP64 logarithm, root and sine, on as
// many SMs as there are tiles) while most SMs have no block of pass A: 64 atoms, k_kick_drift 10.0 us a
// step, the step 48.0 -> 43.1 us.  From 152 tiles on k_kick_drift fills the chip by itself.
__device__ __forceinline__ void draw_ahead(const Bufs& b, int item) {
    const TileAtom ta = tile_of(b, item >> 2);
    const DevSys& S = b.sys[ta.sys];
    const int ia = (item & 3) * 32 + (int)(threadIdx.x & 31), half = (int)(threadIdx.x >> 5);
    if (!S.thermo || ia >= ta.count) return;
    const int i = ta.first + ia;
    uint64_t c[4] = {(uint64_t)b.st[ta.sys].k + 1, (uint64_t)(i - S.off), (uint64_t)S.rng_id, 0ULL};
    philox4x64_10(c, S.seed, 0ULL);
    double z0, z1;
    Noise<double>::pair(half ? c[2] : c[0], half ? c[3] : c[1], z0, z1);
    reinterpret_cast<double2*>(b.xi_next)[2 * (size_t)i + half] = make_double2(z0, half ? 0.0 : z1);
}

template <bool GRAD, bool COMMON>
__global__ void __launch_bounds__(64)
k_edges_d(const __grid_constant__ Bufs b, const __grid_constant__ SWp<double> Pc) {
    dep_wait();
    constexpr unsigned kAll = 0xffffffffu;
    __shared__ EdgesDShared shm[2];
    EdgesDShared& sh = shm[threadIdx.x >> 5];
    if (b.noise_first >= 0 && (int)blockIdx.x >= b.noise_first) {
        draw_ahead(b, (int)blockIdx.x - b.noise_first);
        return;
    }
    const EdgeItem it = edge_item(b);
    const int lg = it.lg, G = 1 << lg, lpa = 5 - lg;
    const TileAtom ta = tile_of(b, it.tile);
    const DevSys& S = b.sys[ta.sys];
    DevState& st = b.st[ta.sys];
    if (S.pot != POT_SW) return;                 // uniform over the block
    const SWp<double>& P = COMMON ? Pc : reinterpret_cast<const SWp<double>*>(b.swc)[S.prm];
    const int lane = threadIdx.x & 31, t = lane & (G - 1);
    const unsigned below = (1u << lane) - 1u;
    const int ia = it.first + ((int)(threadIdx.x >> 5) << lg) + t;   // of the tile
    const int i = ta.first + ia;
    const bool valid = ia < ta.count;
    const double hx = st.h[0], hy = st.h[1], hz = st.h[2];
    const double4* X = reinterpret_cast<const double4*>(b.xs);
    unsigned lo = 0u, hi = 0u;
    if (valid) mark_row(b, i, lane >> lg, lpa, b.lscale[4 * ta.sys], (float)P.rc2, &st.err, lo, hi);
    int ml = __popc(lo) + __popc(hi);            // edges of this lane, then of its atom
    int m = ml, before = 0;                      // before: of the atom's lanes before this one
    for (int o = 16; o >= G; o >>= 1) m += __shfl_xor_sync(kAll, m, o);
    if (__any_sync(kAll, m > kShell)) {          // rare
        if (m > kShell) drop_margin(b, st, P.rc2, i, lane >> lg, lpa, lo, hi);
        m = ml = __popc(lo) + __popc(hi);
        for (int o = 16; o >= G; o >>= 1) m += __shfl_xor_sync(kAll, m, o);
    }
    {
        int inc = ml;                            // inclusive scan over the atom's lanes (stride G)
        for (int o = G; o < 32; o <<= 1) {
            const int y = __shfl_up_sync(kAll, inc, o);
            if (lane >= o) inc += y;
        }
        before = inc - ml;
    }
    int incl = m;                                // edges of atoms 0 .. t
    for (int o = 1; o < G; o <<= 1) {
        const int y = __shfl_up_sync(kAll, incl, o, G);
        if (t >= o) incl += y;
    }
    const int total = __shfl_sync(kAll, incl, G - 1);
    int outside = 0;                             // of the lane's entries, those of the filter's margin
    double red8[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};   // energy, -, virial
    double gth[7] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    double fx = 0.0, fy = 0.0, fz = 0.0, en = 0.0;
    for (int done = 0; done < total;) {
        const bool act = incl - m >= done && incl - done <= kListEdgesD && m > 0;
        const int ma = act ? ml : 0;
        const int mx = __reduce_max_sync(kAll, ma);
        int E = 0;
        {
            const int part = lane >> lg;
            unsigned l = lo, h = hi;
            for (int a = 0; a < mx; ++a) {       // slot by slot: consecutive lanes hold distinct atoms
                const bool on = a < ma;
                const unsigned bal = __ballot_sync(kAll, on);
                if (on) {
                    int k;
                    if (l) { k = __ffs(l) - 1; l &= l - 1u; }
                    else { k = 31 + __ffs(h); h &= h - 1u; }
                    k = 8 * (((k >> 3) << lpa) + part) + (k & 7);
                    const unsigned w = (unsigned)b.nbr[nbr_at(b, i, k)];
                    int j = (int)(w & kIndexMask);
                    if (!NEFE_IN_RANGE(j, b.ntot, &st.err)) j = i;
                    const int e = E + __popc(bal & below), slot = before + a;
                    sh.id[e] = (unsigned)t << kCodeShift | (unsigned)j;
                    sh.slot[e] = (unsigned short)((w >> kCodeShift) << 8 | (unsigned)slot);
                    if (slot < kShell) b.shj[(size_t)i * kShell + slot] = j;
                }
                E += __popc(bal);
            }
        }
        __syncwarp();
        for (int e = lane; e < E; e += 32) {     // edge terms
            const unsigned w = sh.id[e];
            const int code = sh.slot[e] >> 8, ai = i - t + (int)(w >> kCodeShift);
            const double4 xj = X[w & kIndexMask], xi = X[ai];
            const int ox = code % 3 - 1, oy = (code / 3) % 3 - 1, oz = code / 9 - 1;
            const double d[3] = {(xj.x - xi.x) + (ox == 0 ? 0.0 : ox < 0 ? -hx : hx),
                                 (xj.y - xi.y) + (oy == 0 ? 0.0 : oy < 0 ? -hy : hy),
                                 (xj.z - xi.z) + (oz == 0 ? 0.0 : oz < 0 ? -hz : hz)};
            const double none[3] = {0.0, 0.0, 0.0};
            EdgeT<double> q;
            sw_edge_terms<double, double, GRAD>(P, d, none, q);
            if constexpr (GRAD)
                for (int k = 0; k < 5; ++k) gth[k] += 0.5 * q.pg[k];
            sh.v[0][e] = q.ux; sh.v[1][e] = q.uy; sh.v[2][e] = q.uz;
            sh.v[3][e] = q.ir; sh.v[4][e] = q.id; sh.v[5][e] = q.g;
            sh.v[6][e] = q.dphi; sh.v[7][e] = q.r;
            red8[0] = fma(0.5, q.phi, red8[0]);
            if (b.e_atom) reinterpret_cast<double4*>(b.shd)[(size_t)ai * kShell + min(sh.slot[e] & 255, kShell - 1)].w = 0.5 * q.phi;
        }
        __syncwarp();
        MomT<double> M = {};
        int base = 0;
        for (int a = 0; a < mx; ++a) {           // moments
            const bool on = a < ma;
            const unsigned bal = __ballot_sync(kAll, on);
            if (on) {
                const int e = base + __popc(bal & below);
                const double ux = sh.v[0][e], uy = sh.v[1][e], uz = sh.v[2][e];
                // (beyond the cutoff the unit vector is 0: high words, no FP64 comparison)
                outside += ((__double2hiint(ux) | __double2hiint(uy) | __double2hiint(uz)) << 1) == 0 ? 1 : 0;
                mom_add(M, ux, uy, uz, sh.v[5][e]);
            }
            base += __popc(bal);
        }
        double mv[10] = {M.G, M.x, M.y, M.z, M.xx, M.yy, M.zz, M.xy, M.xz, M.yz};
        for (int o = 16; o >= G; o >>= 1)
#pragma unroll
            for (int k = 0; k < 10; ++k) mv[k] += __shfl_xor_sync(kAll, mv[k], o);
        if (lane < G)
#pragma unroll
            for (int k = 0; k < 10; ++k) sh.mom[k][t] = mv[k];
        __syncwarp();
        for (int e = lane; e < E; e += 32) {     // leg forces
            const int te = (int)(sh.id[e] >> kCodeShift), slot = sh.slot[e] & 255, ai = i - t + te;
            MomT<double> Q;
            Q.G = sh.mom[0][te];  Q.x = sh.mom[1][te];  Q.y = sh.mom[2][te];  Q.z = sh.mom[3][te];
            Q.xx = sh.mom[4][te]; Q.yy = sh.mom[5][te]; Q.zz = sh.mom[6][te];
            Q.xy = sh.mom[7][te]; Q.xz = sh.mom[8][te]; Q.yz = sh.mom[9][te];
            const double ux = sh.v[0][e], uy = sh.v[1][e], uz = sh.v[2][e], ir = sh.v[3][e], id = sh.v[4][e], g = sh.v[5][e];
            double lx, ly, lz, s3;
            sw_leg(P, Q, ux, uy, uz, ir, id, g, sh.v[6][e], lx, ly, lz, s3);
            const double gs = g * s3, h = P.eps * P.lam * gs;   // the triplets of edge a, each seen from both its edges
            red8[0] = fma(0.5, h, red8[0]);
            if constexpr (GRAD) {
                const double hi_ = h * id;
                gth[4] = fma(P.gam * hi_, id, gth[4]);
                gth[5] = fma(0.5 * P.eps, gs, gth[5]);
                gth[6] += hi_;
            }
            const double r = sh.v[7][e];
            const double ax = r * lx, ay = r * ly, az = r * lz;
            red8[2] = fma(ux, ax, red8[2]); red8[3] = fma(uy, ay, red8[3]); red8[4] = fma(uz, az, red8[4]);
            red8[5] = fma(ux, ay, fma(uy, ax, red8[5]));
            red8[6] = fma(ux, az, fma(uz, ax, red8[6]));
            red8[7] = fma(uy, az, fma(uz, ay, red8[7]));
            if (slot < kShell) {
                double4* leg = reinterpret_cast<double4*>(b.shd) + (size_t)ai * kShell + slot;
                if (b.e_atom) *leg = mk4(lx, ly, lz, leg->w + 0.5 * h);
                else *leg = mk4(lx, ly, lz, 0.0);
            }
            sh.v[0][e] = lx; sh.v[1][e] = ly; sh.v[2][e] = lz;
        }
        __syncwarp();
        base = 0;
        for (int a = 0; a < mx; ++a) {           // the atoms' own forces
            const bool on = a < ma;
            const unsigned bal = __ballot_sync(kAll, on);
            if (on) {
                const int e = base + __popc(bal & below), slot = min(before + a, kShell - 1);
                fx -= sh.v[0][e]; fy -= sh.v[1][e]; fz -= sh.v[2][e];
                if (b.e_atom) en += reinterpret_cast<const double4*>(b.shd)[(size_t)i * kShell + slot].w;
            }
            base += __popc(bal);
        }
        done = __reduce_max_sync(kAll, act ? incl : 0);
        __syncwarp();
    }
    red8[5] *= 0.5; red8[6] *= 0.5; red8[7] *= 0.5;
    for (int o = 16; o >= G; o >>= 1) {
        outside += __shfl_xor_sync(kAll, outside, o);
        fx += __shfl_xor_sync(kAll, fx, o);
        fy += __shfl_xor_sync(kAll, fy, o);
        fz += __shfl_xor_sync(kAll, fz, o);
        if (b.e_atom) en += __shfl_xor_sync(kAll, en, o);
    }
    if (lane < G && valid) {
        if (m > kShell) atomicOr(&st.err, NEFE_ERR_SHELL_OVERFLOW);
        const int ms = min(m, kShell);
        b.shn[i] = ms | outside << 16;
        if (ms < kShell) b.shj[(size_t)i * kShell + ms] = -1;
        reinterpret_cast<double4*>(b.P)[i] = mk4(fx, fy, fz, en);
    }
    long long* acc = b.acc + (size_t)ta.sys * ACC_N * kSlots;
    const bool engine = b.acc_lo == b.acc;
    block_sum_to_acc<double, 8>(red8, acc, ACC_UINT, &st.err, engine ? acc : b.acc_lo, engine);
    if constexpr (GRAD) block_sum_to_acc<double, 7>(gth, acc, ACC_DTH, &st.err, b.acc_lo);
}

// Force pass B, L lanes per atom:
//   F_SW(i) = P(i) + sum_{j in shell(i)} L_j(i),
// L_j(i) being the leg force that the triplets centred on neighbour j exert on i, stored by
// pass A at the position of i in j's shell (found by scanning j's index list; shells are
// symmetric because both ends compute the same r^2 bit for bit).  Then, in FM_SETUP /
// FM_STEP: Einstein springs, lambda mixing, Langevin force (this step's noise with its
// per-system mean removed), second half kick and the kinetic sums.
template <typename T, int MODE>
__device__ __forceinline__ void finish_atom(const Bufs& b, const DevSys& S, const DevState& st, int i,
                                            const T (&f)[3], T e_i, bool write_e, const T (&pd)[3],
                                            const T (&pv)[3], const T (&pz)[3], const T* s_xm, T (&red)[14],
                                            bool keep, T (&vo)[3], T (&Fo)[3]);
template <typename T>
__device__ __forceinline__ void noise_mean_staged(const DevSys& S, const long long (*xi)[kSlots], T* s_xm);

template <typename T, int MODE, int L>
__global__ void __launch_bounds__(kTile) k_gather(Bufs b) {
    dep_wait();
    using T4 = typename V4<T>::t;
    constexpr int G = kTile / L;
    const int tile = blockIdx.x / L + b.tile_base, part = blockIdx.x % L;
    __shared__ __align__(16) StagedSys sh;
    __shared__ long long s_xi[3][kSlots];
    __shared__ T s_xm[3];
    const TileAtom ta = tile_of(b, tile);
    if (MODE != FM_FORCES) {   // the noise sums' slots, loaded with the descriptors
        const long long* xa = b.acc + (size_t)ta.sys * ACC_N * kSlots + (size_t)ACC_XI * kSlots;
        for (int w = threadIdx.x; w < 3 * kSlots; w += blockDim.x) s_xi[w / kSlots][w % kSlots] = xa[w];
    }
    stage_sys(b, ta.sys, sh);
    __syncthreads();
    const DevSys& S = sh.S;
    const DevState& st = sh.st;
    DevState& gst = b.st[ta.sys];
    if (MODE != FM_FORCES) noise_mean_staged<T>(S, s_xi, s_xm);
    __syncthreads();
    const int lane = threadIdx.x % L, grp = threadIdx.x / L;
    const int lbase = ((threadIdx.x & 31) / L) * L;
    const unsigned gmask = (L == 32) ? 0xffffffffu : (((1u << L) - 1u) << lbase);
    T red[14];
#pragma unroll
    for (int k = 0; k < 14; ++k) red[k] = (T)0;
    const int ia = part * G + grp;
    if (ia < ta.count) {
        const int i = ta.first + ia;
        const size_t N = b.ntot;
        T f[3] = {(T)0, (T)0, (T)0}, e_i = 0;
        // the epilogue's own-atom operands are loaded first, so their latency overlaps the gather
        T pd[3] = {(T)0, (T)0, (T)0}, pv[3] = {(T)0, (T)0, (T)0}, pz[3] = {(T)0, (T)0, (T)0};
        if (MODE != FM_FORCES && lane == 0) {
            if (S.springs) {
                const T4 d0 = reinterpret_cast<const T4*>(b.sd0)[i];
                const T* DH = reinterpret_cast<const T*>(b.dhi);
                const T* DL = reinterpret_cast<const T*>(b.dlo);
                pd[0] = d0.x; pd[1] = d0.y; pd[2] = d0.z;
                for (int k = 0; k < 3; ++k) {
                    pd[k] += DH[k * N + i];
                    if constexpr (sizeof(T) == 4) pd[k] += DL[k * N + i];
                }
            }
            const T* V = reinterpret_cast<const T*>(b.v);
            pv[0] = V[i]; pv[1] = V[N + i]; pv[2] = V[2 * N + i];
            if (S.thermo) {
                const T4 z = reinterpret_cast<const T4*>(b.xi)[i];
                pz[0] = z.x; pz[1] = z.y; pz[2] = z.z;
            }
        }
        if (S.pot == POT_SW) {
            const T4* Fl = reinterpret_cast<const T4*>(b.shd);
            const int m = b.shn[i] & 0xffff;     // (FP64: with the margin's entries, see k_edges_d)
            // NB shell entries per lane in flight: neighbour index, the first 8 entries of the
            // neighbour's index list (one 32-byte sector), then the leg force
            constexpr int NB = L >= 2 ? 1 : 2;
            for (int base = 0; base < m; base += NB * L) {
                int jj[NB], pos[NB];
                int4 q0[NB], q1[NB];
                if constexpr (NB == 2 && L == 1) {   // both entries with one 8-byte load (rows are 128 bytes)
                    const int2 j2 = *reinterpret_cast<const int2*>(b.shj + (size_t)i * kShell + base);
                    jj[0] = j2.x;
                    jj[NB - 1] = base + 1 < m ? j2.y : -1;
                } else {
#pragma unroll
                    for (int u = 0; u < NB; ++u) {
                        const int a = base + u * L + lane;
                        jj[u] = a < m ? b.shj[(size_t)i * kShell + a] : -1;
                    }
                }
#pragma unroll
                for (int u = 0; u < NB; ++u)
                    if (jj[u] >= 0 && !NEFE_IN_RANGE(jj[u], b.ntot, &gst.err)) jj[u] = -1;
#pragma unroll
                for (int u = 0; u < NB; ++u) {
                    if (jj[u] >= 0) {
                        const int4* Sq = reinterpret_cast<const int4*>(b.shj + (size_t)jj[u] * kShell);
                        q0[u] = Sq[0];
                        q1[u] = Sq[1];
                    }
                }
#pragma unroll
                for (int u = 0; u < NB; ++u) {
                    pos[u] = -1;
                    if (jj[u] < 0) continue;
                    const int w8[8] = {q0[u].x, q0[u].y, q0[u].z, q0[u].w, q1[u].x, q1[u].y, q1[u].z, q1[u].w};
                    bool ended = false;
#pragma unroll
                    for (int t = 0; t < 8; ++t) {
                        if (!ended && pos[u] < 0) {
                            if (w8[t] == i) pos[u] = t;
                            else if (w8[t] < 0) ended = true;
                        }
                    }
                    if (pos[u] < 0 && !ended) {          // i beyond the first 8 entries of j's shell
                        const int* Sj = b.shj + (size_t)jj[u] * kShell;
                        for (int t = 8; t < kShell; ++t) {
                            const int q = Sj[t];
                            if (q == i) { pos[u] = t; break; }
                            if (q < 0) break;
                        }
                    }
                }
                T4 lf[NB];
#pragma unroll
                for (int u = 0; u < NB; ++u)
                    if (pos[u] >= 0) lf[u] = Fl[(size_t)jj[u] * kShell + pos[u]];
#pragma unroll
                for (int u = 0; u < NB; ++u)
                    if (pos[u] >= 0) { f[0] += lf[u].x; f[1] += lf[u].y; f[2] += lf[u].z; }
            }
#pragma unroll
            for (int o = L / 2; o > 0; o >>= 1) {
                f[0] += __shfl_xor_sync(gmask, f[0], o);
                f[1] += __shfl_xor_sync(gmask, f[1], o);
                f[2] += __shfl_xor_sync(gmask, f[2], o);
            }
            const T4* Pa = reinterpret_cast<const T4*>(b.P);
            const T4 p = Pa[i];
            f[0] += p.x; f[1] += p.y; f[2] += p.z; e_i = p.w;
            if (sizeof(T) == 4 && lane == 0) {   // (FP64: summed by pass A)
                const T4 wa = Pa[b.ntot + 2 * (size_t)i], wb = Pa[b.ntot + 2 * (size_t)i + 1];
                red[0] = e_i;
                red[2] = wa.x; red[3] = wa.y; red[4] = wa.z; red[5] = wa.w; red[6] = wb.x; red[7] = wb.y;
            }
        }
        T vo[3], Fo[3];
        if (lane == 0) finish_atom<T, MODE>(b, S, st, i, f, e_i, true, pd, pv, pz, s_xm, red, false, vo, Fo);
    }
    block_sum_to_acc<T, 14>(red, b.acc + (size_t)ta.sys * ACC_N * kSlots, ACC_UINT, &gst.err);
}

// The epilogue of force pass B for atom i with SW (or zero) force f: the stateless output, or
// Einstein springs / UF force, lambda mixing, Langevin force with the per-system mean of this
// step's noise removed, second half kick, total force for the next step and the kinetic sums.
// pd: spring offset x - r0; pv: velocity; pz: noise of the step; s_xm: the per-system noise mean.
// keep: the velocity and total force are returned in vo, Fo instead of being stored (the caller
// goes on to the next step's kick and drift).
template <typename T, int MODE>
__device__ __forceinline__ void finish_atom(const Bufs& b, const DevSys& S, const DevState& st, int i,
                                            const T (&f)[3], T e_i, bool write_e, const T (&pd)[3],
                                            const T (&pv)[3], const T (&pz)[3], const T* s_xm, T (&red)[14],
                                            bool keep, T (&vo)[3], T (&Fo)[3]) {
    using T4 = typename V4<T>::t;
    const size_t N = b.ntot;
            if (MODE == FM_FORCES) {
                b.f_out[i] = (double)f[0]; b.f_out[N + i] = (double)f[1]; b.f_out[2 * N + i] = (double)f[2];
                if (b.e_atom && write_e) b.e_atom[i] = (double)e_i;
            } else {
                T fint[3] = {f[0], f[1], f[2]}, fe[3] = {(T)0, (T)0, (T)0};
                T u_int = 0, u_ref = 0;
                if (S.springs) {
                    const T d[3] = {pd[0], pd[1], pd[2]};
                    const T d2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
                    if (S.pot == POT_EINSTEIN) {
                        const T k_i = pick<T>(S.k_int, S.kint_f);
                        u_int = (T)0.5 * k_i * d2;
                        for (int k = 0; k < 3; ++k) fint[k] = -k_i * d[k];
                    }
                    const T k_e = pick<T>(S.k_E, S.kE_f);
                    u_ref = (T)0.5 * k_e * d2;
                    for (int k = 0; k < 3; ++k) fe[k] = -k_e * d[k];
                }
                if (S.uf_mode != UF_NONE) {     // UF force of this step (its energy is summed by k_uf)
                    const T4 fu = reinterpret_cast<const T4*>(b.uf_F)[i];
                    T* dst = S.uf_mode == UF_INT ? fint : fe;
                    dst[0] = fu.x; dst[1] = fu.y; dst[2] = fu.z;
                }
                T* V = reinterpret_cast<T*>(b.v);
                T v[3] = {pv[0], pv[1], pv[2]};
                const T si = pick<T>(st.scale_int, st.scale_int_f), se = pick<T>(st.scale_E, st.scale_E_f);
                T F[3];
                for (int k = 0; k < 3; ++k) F[k] = si * fint[k] + se * fe[k];
                if (S.thermo) {
                    const T zz[3] = {pz[0], pz[1], pz[2]};
                    const T amp = pick<T>(S.amp, S.amp_f), gam = pick<T>(S.gam, S.gam_f);
                    for (int k = 0; k < 3; ++k) F[k] += -gam * v[k] + amp * (zz[k] - s_xm[k]);
                }
                if (MODE == FM_STEP) {
                    const T ck = pick<T>(S.ckick, S.ckick_f);
                    for (int k = 0; k < 3; ++k) {
                        v[k] += ck * F[k];
                        if (!keep) V[k * N + i] = v[k];
                    }
                }
                for (int k = 0; k < 3; ++k) { vo[k] = v[k]; Fo[k] = F[k]; }
                if (!keep) reinterpret_cast<T4*>(b.F)[i] = mk4(F[0], F[1], F[2], (T)0);
                const T me = pick<T>(S.mass_e, S.mass_f);
                red[0] += u_int;
                red[1] = u_ref;
                red[8] = me * v[0] * v[0];
                red[9] = me * v[1] * v[1];
                red[10] = me * v[2] * v[2];
                red[11] = me * v[0] * v[1];
                red[12] = me * v[0] * v[2];
                red[13] = me * v[1] * v[2];
            }
}

// Per-system mean of this step's thermostat noise (the "zero yes" removal), from the
// fixed-point sums of k_kick_drift, into s_xm[3]: xi holds their slots, already copied to shared memory
// (3 x kSlots).  Threads 0..2 write; the caller syncs.
template <typename T>
__device__ __forceinline__ void noise_mean_staged(const DevSys& S, const long long (*xi)[kSlots], T* s_xm) {
    if (threadIdx.x < 3) {
        long long sum = 0;
        for (int sl = 0; sl < kSlots; ++sl) sum += xi[threadIdx.x][sl];
        if constexpr (sizeof(T) == 4) {
            const float hi = (float)(int)(sum >> 32);
            const float lo = (float)(unsigned)(sum & 0xffffffffLL) * 0x1p-32f;
            s_xm[threadIdx.x] = (hi + lo) * S.inv_n_f;
        } else {
            s_xm[threadIdx.x] = (T)((double)sum / kFix / (double)S.n);
        }
    }
}

// Force pass B of the scatter form: one thread per atom reads and clears the atom's force
// accumulator (the pair, own-triplet and leg forces pass A added) and runs the epilogue.  The
// SW energy and virial were summed by pass A.
// fuse (FM_STEP, systems without a barostat): the epilogue goes straight on to the next step's
// first half kick, drift, mirror, displacement test and thermostat noise -- the work of
// k_kick_drift, which then skips these systems.  Nothing between the two reads or changes what
// that work uses (no barostat: the box, drift factors and rebuild threshold stay as they are),
// and the operations are the same ones, so the trajectory is bit for bit that of the unfused
// sequence.  The force of the step is not stored (the next half kick consumed it); the noise
// sums go to ACC_XIN and the rebuild flag to rebuild_next, which the next k_group moves into
// place.  The last step of every launch sequence runs unfused, so the state between calls is
// the usual one (positions and velocities at a full step).
// FP32: nine blocks an SM (56 registers, one spilled on the rare path of the large terms); left to itself the
// kernel takes 61 and holds eight: 128 x 8000 atoms 82.75 -> 82.15 ms a pass, 64 pairs 64.4 -> 63.95.
template <typename T, int MODE>
__global__ void __launch_bounds__(kTile, sizeof(T) == 4 ? 9 : 1) k_finish(Bufs b, int fuse) {
    dep_wait();
    using T4 = typename V4<T>::t;
    const int tile = blockIdx.x + b.tile_base;
    __shared__ __align__(16) StagedSys sh;
    __shared__ long long s_xi[3][kSlots];
    __shared__ T s_xm[3];
    const TileAtom ta = tile_of(b, tile);
    const bool valid = (int)threadIdx.x < ta.count;
    const int i = ta.first + threadIdx.x;
    const size_t N = b.ntot;
    // The atom's operands and the system's descriptors are loaded together, before the first is
    // looked at (nothing else hides this kernel's latency; what a system does not use is loaded all
    // the same and ignored: arrays of every context).
    int4* a4 = reinterpret_cast<int4*>(b.lacc) + i;
    int4 q = make_int4(0, 0, 0, 0), fb = q;
    T4 d0 = mk4((T)0, (T)0, (T)0, (T)0), z = d0, xa = d0;
    T dh[3] = {(T)0, (T)0, (T)0}, dl[3] = {(T)0, (T)0, (T)0}, pv[3] = {(T)0, (T)0, (T)0};
    BoxMove bm{};
    if (valid) {
        q = *a4;
        if (MODE != FM_FORCES) {
            const T* DH = reinterpret_cast<const T*>(b.dhi);
            const T* DL = reinterpret_cast<const T*>(b.dlo);
            const T* V = reinterpret_cast<const T*>(b.v);
            d0 = reinterpret_cast<const T4*>(b.sd0)[i];
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                dh[k] = DH[k * N + i];
                if constexpr (sizeof(T) == 4) dl[k] = DL[k * N + i];
                pv[k] = V[k * N + i];
            }
            z = reinterpret_cast<const T4*>(b.xi)[i];
            if (MODE == FM_STEP && fuse) {
                if (b.want_xf) bm = box_move(b, ta.sys);
                if (b.want_xs) xa = reinterpret_cast<const T4*>(b.xa)[i];   // (no barostat: the box never moves)
                if (b.want_xf) fb = b.xfb[i];
            }
        }
    }
    const int big = b.hi_flag ? b.hi_flag[tile] : 0;                        // large terms were split
    if (MODE != FM_FORCES) {   // the noise sums' slots, loaded with the descriptors
        const long long* xs = b.acc + (size_t)ta.sys * ACC_N * kSlots + (size_t)ACC_XI * kSlots;
        for (int w = threadIdx.x; w < 3 * kSlots; w += blockDim.x) s_xi[w / kSlots][w % kSlots] = xs[w];
    }
    stage_sys(b, ta.sys, sh);
    __syncthreads();
    const DevSys& S = sh.S;
    const DevState& st = sh.st;
    DevState& gst = b.st[ta.sys];
    if (MODE != FM_FORCES) noise_mean_staged<T>(S, s_xi, s_xm);
    __syncthreads();
    if (big != 0 && threadIdx.x == 0) b.hi_flag[tile] = 0;            // every thread has read it
    const bool fz = MODE == FM_STEP && fuse && S.baro == BARO_NONE;   // uniform over the block
    T red[14];
#pragma unroll
    for (int k = 0; k < 14; ++k) red[k] = (T)0;
    T zn[3] = {(T)0, (T)0, (T)0};
    if (valid) {
        const bool sw = S.pot == POT_SW;
        if (sw) *a4 = make_int4(0, 0, 0, 0);
        else q = make_int4(0, 0, 0, 0);
        const T pd[3] = {d0.x + dh[0] + dl[0], d0.y + dh[1] + dl[1], d0.z + dh[2] + dl[2]};
        const T pz[3] = {z.x, z.y, z.z};
        const T inv = (T)S.leg_unit_f;
        const int3 fq = force_of_acc(q);
        T f[3] = {(T)fq.x * inv, (T)fq.y * inv, (T)fq.z * inv};
        if (sw && big != 0) {
            long long* h3 = b.lacc_hi + 3 * (size_t)i;
            const T coarse = (T)(kLegCoarse * kLegScale) * inv;
#pragma unroll
            for (int k = 0; k < 3; ++k) {
                const long long h = h3[k];
                h3[k] = 0;
                if (h == (long long)(int)h) f[k] += coarse * (T)(int)h;
                else if (h >= kLegLost || h <= -kLegLost) f[k] = (T)NAN;
                else f[k] += coarse * (T)h;
            }
        }
        T vo[3], Fo[3];
        finish_atom<T, MODE>(b, S, st, i, f, (T)0, false, pd, pv, pz, s_xm, red, fz, vo, Fo);
        if (fz) {
            // the next step's first half kick (the force of this step, Langevin term included)
            T* V = reinterpret_cast<T*>(b.v);
            const T ck = pick<T>(S.ckick, S.ckick_f);
            T vk[3];
            for (int k = 0; k < 3; ++k) {
                vk[k] = fma_rn(ck, Fo[k], vo[k]);
                V[k * N + i] = vk[k];
            }
            drift_atom<T>(b, S, st, bm, i, xa, fb, vk, true, dh, dl, 0, &gst.rebuild_next,
                          b.any_rebuild ? b.any_rebuild + 1 : nullptr, (unsigned long long)st.k + 1ULL,
                          zn);
        }
    }
    block_sum_to_acc<T, 14>(red, b.acc + (size_t)ta.sys * ACC_N * kSlots, ACC_UINT, &gst.err);
    if (fz) block_sum_to_acc<T, 3>(zn, b.acc + (size_t)ta.sys * ACC_N * kSlots, ACC_XIN, &gst.err);
}

// FP64 positions and velocities for output, and replacement from FP64 input.
template <typename T>
__global__ void __launch_bounds__(kTile) k_materialize(Bufs b, double* x, double* v) {
    dep_wait();
    const TileAtom ta = tile_of(b, blockIdx.x);
    if ((int)threadIdx.x >= ta.count) return;
    const int i = ta.first + threadIdx.x;
    const size_t N = b.ntot;
    const T* DH = reinterpret_cast<const T*>(b.dhi);
    const T* DL = reinterpret_cast<const T*>(b.dlo);
    const T* V = reinterpret_cast<const T*>(b.v);
    for (int k = 0; k < 3; ++k) {
        if (x) {
            double d = (double)DH[k * N + i];
            if constexpr (sizeof(T) == 4) d += (double)DL[k * N + i];
            x[k * N + i] = b.x[k * N + i] + d;
        }
        if (v) v[k * N + i] = (double)V[k * N + i];
    }
}

template <typename T>
__global__ void __launch_bounds__(kTile) k_inject(Bufs b, const double* x, const double* v) {
    dep_wait();
    const TileAtom ta = tile_of(b, blockIdx.x);
    if ((int)threadIdx.x >= ta.count) return;
    const int i = ta.first + threadIdx.x;
    const size_t N = b.ntot;
    T* DH = reinterpret_cast<T*>(b.dhi);
    T* DL = reinterpret_cast<T*>(b.dlo);
    T* V = reinterpret_cast<T*>(b.v);
    for (int k = 0; k < 3; ++k) {
        if (x) {
            b.x[k * N + i] = x[k * N + i];
            DH[k * N + i] = (T)0;
            if constexpr (sizeof(T) == 4) DL[k * N + i] = (T)0;
        }
        if (v) V[k * N + i] = (T)v[k * N + i];
    }
}

// ------------------------------------------------------------------------------------
// Per-group update (one 128-thread block per system or dCCI pair).
// ------------------------------------------------------------------------------------
__device__ double sched_lambda(const DevSys& S, long long k) {
    double tau = (double)k / (double)S.nsched;
    if (tau > 1.0) tau = 1.0;
    if (S.direction < 0) tau = 1.0 - tau;
    switch (S.sched) {
        case SCHED_FL: {
            const double t2 = tau * tau, t4 = t2 * t2;
            return t4 * tau * (70.0 * t4 - 315.0 * t2 * tau + 540.0 * t2 - 420.0 * tau + 126.0);
        }
        case SCHED_RS: return 1.0 / (1.0 + tau * (1.0 / S.lam_f - 1.0));
        case SCHED_AS: return S.p0 + (S.p1 - S.p0) * tau;
        default: return S.lam0;
    }
}

__device__ __forceinline__ void force_scales(const DevSys& S, DevState& st) {
    double s_int, s_e;
    if (S.sched == SCHED_FL) { s_int = 1.0 - st.lam; s_e = st.lam; }
    else if (S.sched == SCHED_RS || S.pair >= 0) { s_int = st.lam; s_e = 0.0; }
    else if (S.sched == SCHED_NONE) { s_int = S.lam0; s_e = 0.0; }
    else { s_int = 1.0; s_e = 0.0; }
    st.scale_int = s_int;
    st.scale_E = s_e;
    st.scale_int_f = (float)s_int;
    st.scale_E_f = (float)s_e;
}

__device__ __forceinline__ double target_pressure(const DevSys& S, const DevState& st) {
    if (S.sched == SCHED_RS) return st.lam * S.p_phys;
    if (S.sched == SCHED_AS) return st.lam;
    if (S.pair >= 0) return st.p_tgt;
    return S.p_ext;
}

// The per-group update runs on one warp per member, its lanes in step: what is one value per axis or
// per stress component is one lane's, the rest is computed by every lane alike (a dependent FP64
// operation costs some 90 cycles here, so what counts is the length of the chain, not the lanes).
//
// Observation of the step just finished: P, V, dH/dlambda, H.
__device__ __forceinline__ void observe(const DevSys& S, DevState& st, int lane) {
    const double V = st.box[0] * st.box[1] * st.box[2];
    const double K = 0.5 * (st.kt[0] + st.kt[1] + st.kt[2]);
    if (lane < 6) st.P[lane] = (st.kt[lane] + st.scale_int * st.vir[lane]) / V;
    double dhdl = 0.0, H;
    if (S.sched == SCHED_FL) {
        dhdl = st.u_ref - st.u_int;
        H = K + (1.0 - st.lam) * st.u_int + st.lam * st.u_ref;
    } else if (S.sched == SCHED_RS) {
        dhdl = st.u_int + S.p_phys * V;
        H = K + st.lam * st.u_int + st.lam * S.p_phys * V;
    } else if (S.sched == SCHED_AS) {
        dhdl = V;
        H = K + st.u_int + st.lam * V;
    } else {
        H = K + st.scale_int * st.u_int + (S.baro != BARO_NONE ? target_pressure(S, st) * V : 0.0);
    }
    __syncwarp();
    if (lane == 0) {
        st.V = V;
        st.dHdl = dhdl;
        st.H = H;
    }
    __syncwarp();
}

// Running sums, trace row, and the barostat's kick (one axis per lane).
__device__ __forceinline__ void record_and_kick(const DevSys& S, DevState& st, double dt, double* trace, int lane) {
    const double P = (st.P[0] + st.P[1] + st.P[2]) / 3.0;
    if (lane < 5) st.sums[lane] += lane == 0 ? st.H : lane == 1 ? st.dHdl : lane == 2 ? P : lane == 3 ? st.V : 1.0;
    if (S.trace_every > 0 && S.trace_cap > 0 && st.k % S.trace_every == 0 && lane == 0) {
        double* r = trace + (S.trace_off + st.trace_n % S.trace_cap) * 9;
        r[0] = (double)st.k; r[1] = st.lam; r[2] = st.W; r[3] = st.dHdl; r[4] = st.u_int;
        r[5] = st.V; r[6] = P * kEvA3ToGPa; r[7] = target_pressure(S, st) * kEvA3ToGPa;
        r[8] = (st.kt[0] + st.kt[1] + st.kt[2]) / ((3.0 * S.n - 3.0) * kB);
        st.trace_n += 1;
    }
    if (S.baro != BARO_NONE && lane < 3) {
        const double ptgt = target_pressure(S, st);
        // S.baro_c = dt / Q_b, Q_b = (N + 1) kB T tau_P^2
        if (S.baro == BARO_ISO) st.eta[lane] += S.baro_c * (3.0 * st.V * (P - ptgt));
        else st.eta[lane] += S.baro_c * (st.V * (st.P[lane] - ptgt));
    }
    __syncwarp();
}

// This step's force scales, drift factors, box and list threshold (one axis per lane).
__device__ __forceinline__ void prepare_step(const Bufs& b, int s, const DevSys& S, DevState& st, int lane) {
    if (lane == 0) force_scales(S, st);
    double rel = 0.0;
    bool scaled = false, hm = false;
    const bool moved = st.hmoved != 0;
    const int k = lane < 3 ? lane : 0;
    const double z = st.eta[k] * b.dt;
    double sk = 1.0, ph = 1.0;
    if (z != 0.0) {
        const double em = expm1(z);
        sk = 1.0 + em;
        ph = em / z;
    }
    scaled = __any_sync(0xffffffffu, sk != 1.0);
    // With no axis scaled and the cell edge still the one of the last build, the box, h = box /
    // ncell, h / hb = 1 and their FP32 copies are what they were: the FP64 divisions are skipped.
    double box = st.box[k], h = 0.0, ratio = 1.0;
    if (scaled || moved) {
        box *= sk;
        h = box / (double)st.ncell[k];
        ratio = h / st.hb[k];
        rel = fabs(ratio - 1.0);
        hm = __any_sync(0xffffffffu, h != st.hb[k]);
        rel = fmax(rel, fmax(__shfl_sync(0xffffffffu, rel, 1), __shfl_sync(0xffffffffu, rel, 2)));   // (lane 0's use)
    }
    __syncwarp();
    if (lane < 3) {
        st.s[lane] = sk;
        st.phi[lane] = ph;
        st.phi_f[lane] = (float)ph;
        st.sm1_f[lane] = (float)(sk - 1.0);
        if (scaled || moved) {
            st.box[lane] = box;
            st.h[lane] = h;
            st.h_f[lane] = (float)h;
            st.hb_f[lane] = (float)st.hb[lane];
            st.rho_f[lane] = (float)ratio;
            if (b.lscale) scale_axis(b, s, lane, box, hm ? 1.0 - ratio : 0.0);
        }
    }
    if (lane == 0) {
        if (scaled || moved) st.hmoved = hm ? 1 : 0;
        st.scaled = scaled ? 1 : 0;
        const double thr = 0.5 * (S.skin - rel * S.rcs);
        st.thr2 = thr > 0.0 ? thr * thr : -1.0;
        st.thr2_f = (float)st.thr2;
    }
    __syncwarp();
}

// carry (mode 1): the previous step's epilogue already kicked and moved the systems without a
// barostat and drew their noise for this step (k_finish with fuse): their next-step noise sums
// (ACC_XIN) become this step's (ACC_XI) and rebuild_next becomes rebuild, instead of both being
// cleared.
// One block per group.  The members' descriptors and states (and the pair's state) are updated in
// shared memory; the fixed-point sums are read while they arrive.  Warp m updates member m (see
// observe), warp 2 meanwhile what depends on the step counter alone (the schedule's next lambda, the
// controlled variable of a pair).  Before, one thread did all of it: 9.3 -> 6.5 us for one system,
// 16.5 -> 8.4 us for 12 and 35 -> 14 us for 64 pairs under barostats.
struct GroupShared {
    StagedSys m[2];
    DevPair pr;
    double next[3];      // lambda (schedule); T or p at this step and the next (pair)
};
__global__ void __launch_bounds__(kTile) k_group(Bufs b, const DevGroup* groups, int mode, int carry) {
    dep_wait();
    const DevGroup gr = groups[blockIdx.x];
    const int nm = gr.b >= 0 ? 2 : 1;
    __shared__ __align__(16) GroupShared sh;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int mine = warp == 1 ? gr.b : gr.a;    // the member of warps 0 and 1
    // slot sums (fixed order: deterministic), in flight together with the descriptors; lane 16 + a takes the
    // remainders of sum a where pass A keeps them (FP64)
    double sum = 0.0;
    const int a_lo = lane - 16;
    const bool rest = b.acc_lo && a_lo >= 0 && a_lo < ACC_KT && a_lo != ACC_UREF;
    if (mode != 0 && warp < nm && (lane < ACC_XI || rest))
        sum = (double)slot_sum(b.acc + ((size_t)mine * ACC_N + (rest ? engine_lo_row(a_lo) : lane)) * kSlots) *
              (rest ? 0x1p-40 : 1.0 / kFix);
    for (int mi = 0; mi < nm; ++mi) {
        StagedSys& m = sh.m[mi];
        stage_sys(b, mi == 0 ? gr.a : gr.b, m);
    }
    if (gr.pair >= 0) {
        constexpr int wp = (int)(sizeof(DevPair) / 4);
        const uint32_t* gp = reinterpret_cast<const uint32_t*>(b.pairs + gr.pair);
        for (int w = threadIdx.x; w < wp; w += blockDim.x) reinterpret_cast<uint32_t*>(&sh.pr)[w] = gp[w];
    }
    __syncthreads();
    if (warp < nm && mode != 0) {
        DevState& st = sh.m[warp].st;
        sum += __shfl_down_sync(0xffffffffu, sum, 16);
        if (lane == ACC_UINT) st.u_int = sum;
        else if (lane == ACC_UREF) st.u_ref = sum;
        else if (lane < ACC_KT) st.vir[lane - ACC_VIR] = sum;
        else if (lane < ACC_XI) st.kt[lane - ACC_KT] = sum;
        __syncwarp();
        observe(sh.m[warp].S, st, lane);
        if (mode == 1) record_and_kick(sh.m[warp].S, st, b.dt, b.trace, lane);
    } else if (warp == 2 && mode == 1 && lane < 2) {
        if (gr.pair >= 0) {                      // lane 0: tau of this step, lane 1: of the next
            const DevPair& pr = sh.pr;
            const double tau = fmin((double)(pr.k + lane) / (double)pr.nsteps, 1.0);
            sh.next[1 + lane] = pr.frm + (pr.to - pr.frm) * tau;
        } else if (lane == 0 && sh.m[0].S.sched != SCHED_NONE) {
            sh.next[0] = sched_lambda(sh.m[0].S, sh.m[0].st.k + 1);
        }
    }
    __syncthreads();
    if (mode == 0) {
        if (warp < nm) {
            const DevSys& S = sh.m[warp].S;
            DevState& st = sh.m[warp].st;
            if (lane == 0) {
                if (S.pair >= 0) {               // a paired system's group is its pair
                    st.lam = 1.0;
                    st.p_tgt = sh.pr.ps;
                } else if (S.sched != SCHED_NONE) {
                    st.lam = sched_lambda(S, st.k);
                }
                force_scales(S, st);
                for (int k = 0; k < 3; ++k) {
                    st.s[k] = 1.0; st.phi[k] = 1.0; st.phi_f[k] = 1.0f; st.sm1_f[k] = 0.0f;
                }
                st.scaled = 0;
                scale_of_box(b, mine, st);
            }
        }
    } else if (mode == 1) {
        if (threadIdx.x == 0) {
            if (gr.pair >= 0) {
                DevPair& pr = sh.pr;
                DevState& A = sh.m[0].st;
                DevState& B = sh.m[1].st;
                const double du = A.u_int / sh.m[0].S.n - B.u_int / sh.m[1].S.n;
                const double dv = A.V / sh.m[0].S.n - B.V / sh.m[1].S.n;
                double lam_next, ps_next;
                if (pr.mode == 0) {
                    lam_next = pr.frm / sh.next[2];
                    if (fabs(dv) < 1e-6) {
                        pr.err |= NEFE_ERR_DEGEN;
                        lam_next = pr.lam; ps_next = pr.ps;
                    } else {
                        ps_next = pr.ps - (lam_next - pr.lam) * (du / dv);
                    }
                } else {
                    const double p0 = sh.next[1], p1 = sh.next[2];
                    if (fabs(du) < 1e-12) {
                        pr.err |= NEFE_ERR_DEGEN;
                        lam_next = pr.lam; ps_next = pr.ps;
                    } else {
                        const double g = dv / du;
                        lam_next = pr.lam * (1.0 + p0 * g) / (1.0 + p1 * g);
                        ps_next = lam_next * p1;
                    }
                }
                pr.lam = lam_next;
                pr.ps = ps_next;
                pr.k += 1;
                A.lam = B.lam = lam_next;
                A.p_tgt = B.p_tgt = ps_next;
                if (pr.err) { A.err |= pr.err; B.err |= pr.err; }
            } else if (sh.m[0].S.sched != SCHED_NONE) {
                DevState& st = sh.m[0].st;
                st.W += st.dHdl * (sh.next[0] - st.lam);
                st.lam = sh.next[0];
            }
        }
        __syncthreads();
        if (warp < nm) {
            DevState& st = sh.m[warp].st;
            prepare_step(b, mine, sh.m[warp].S, st, lane);
            if (lane == 0) {
                st.rebuild = (carry && sh.m[warp].S.baro == BARO_NONE) ? st.rebuild_next : 0;
                st.rebuild_next = 0;
                st.k += 1;
            }
        }
    }
    __syncthreads();
    for (int mi = 0; mi < nm; ++mi) {
        constexpr int wt = (int)(sizeof(DevState) / 4);
        uint32_t* gt = reinterpret_cast<uint32_t*>(b.st + (mi == 0 ? gr.a : gr.b));
        const uint32_t* dt = reinterpret_cast<const uint32_t*>(&sh.m[mi].st);
        for (int w = threadIdx.x; w < wt; w += blockDim.x) gt[w] = dt[w];
    }
    if (gr.pair >= 0) {
        constexpr int wp = (int)(sizeof(DevPair) / 4);
        uint32_t* gp = reinterpret_cast<uint32_t*>(b.pairs + gr.pair);
        for (int w = threadIdx.x; w < wp; w += blockDim.x) gp[w] = reinterpret_cast<const uint32_t*>(&sh.pr)[w];
    }
    // the context-wide flag word: this step's flags start from the fused epilogue's (carry) or
    // from none; the next step's word is cleared (block 0 only; no other block touches it)
    if (mode == 1 && b.any_rebuild && blockIdx.x == 0 && threadIdx.x == 0) {
        b.any_rebuild[0] = carry ? b.any_rebuild[1] : 0;
        b.any_rebuild[1] = 0;
    }
    if (mode != 2) {
        for (int mi = 0; mi < nm; ++mi) {
            long long* acc = b.acc + (size_t)(mi == 0 ? gr.a : gr.b) * ACC_N * kSlots;
            const bool moved = mode == 1 && carry && sh.m[mi].S.baro == BARO_NONE;
            for (int t = threadIdx.x; t < ACC_N * kSlots; t += blockDim.x) {
                const int a = t / kSlots;
                long long v = 0;
                if (moved && a >= ACC_XI && a < ACC_XI + 3) v = acc[t + (ACC_XIN - ACC_XI) * kSlots];
                if (a < ACC_XIN) acc[t] = v;
            }
            __syncthreads();   // ACC_XIN is read above before it is cleared
            for (int t = threadIdx.x; t < 3 * kSlots; t += blockDim.x) acc[ACC_XIN * kSlots + t] = 0;
        }
    }
}

__global__ void k_noise(unsigned long long seed, unsigned long long sys, unsigned long long step, int n,
                        int prec, double* xi) {
    dep_wait();
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    if (prec == NEFE_FP64) {
        double z[3];
        Noise<double>::xi3(seed, sys, step, (uint64_t)i, z);
        for (int k = 0; k < 3; ++k) xi[3 * i + k] = z[k];
    } else {
        float z[3];
        Noise<float>::xi3(seed, sys, step, (uint64_t)i, z);
        for (int k = 0; k < 3; ++k) xi[3 * i + k] = (double)z[k];
    }
}

// (n,3) row-major <-> SoA with stride n.
__global__ void k_aos_to_soa(const double* __restrict__ a, double* __restrict__ s, int n) {
    dep_wait();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= 3 * n) return;
    const int i = t / 3, k = t % 3;
    s[(size_t)k * n + i] = a[t];
}
__global__ void k_soa_to_aos(const double* __restrict__ s, double* __restrict__ a, int n) {
    dep_wait();
    const int t = blockIdx.x * blockDim.x + threadIdx.x;
    if (t >= 3 * n) return;
    const int i = t / 3, k = t % 3;
    a[t] = s[(size_t)k * n + i];
}

// Sum a of a stateless call: slots and remainders (stateless calls hold both, one after the other).
__device__ __forceinline__ double decoded(const long long* acc, int a) {
    const long long* lo = acc + (size_t)ACC_N * kSlots;
    return (double)slot_sum(acc + (size_t)a * kSlots) / kFix + (double)slot_sum(lo + (size_t)a * kSlots) * 0x1p-40;
}
// (NaN where a block's sum was out of range or not finite and is missing: err, or NULL)
__global__ void k_decode_ev(const long long* acc, double* out7, const unsigned* err) {
    dep_wait();
    const int t = threadIdx.x;
    if (t >= 7) return;
    const int a = t == 0 ? ACC_UINT : ACC_VIR + (t - 1);
    out7[t] = err && (*err & NEFE_ERR_NAN) ? NAN : decoded(acc, a);
}

// ------------------------------------------------------------------------------------
// Launchers
// ------------------------------------------------------------------------------------
bool lanes_supported(int lanes) {
    return lanes == 0 || lanes == 1 || lanes == 4 || lanes == 8 || lanes == 16 || lanes == 32;
}

// With a worklist (engine) the per-tile rebuild kernels get a bounded grid and walk the
// flagged tiles; without one (stateless calls) they cover every tile.
static int rebuild_grid(const Bufs& b, int items) {
    return b.rtiles ? (items < kRebuildBlocks ? items : kRebuildBlocks) : items;
}

// Blocks of the list builds: a warp for every cell there can be (ncells_host), up to kRebuildBlocks; on a
// step without a rebuild the launch costs what its blocks cost to start (1216 blocks 2.7 us).
static int list_grid(const Bufs& b, int ntiles) {
    const int most = b.ncells_host > 0 ? (b.ncells_host + kTile / 32 - 1) / (kTile / 32) : ntiles * 8;
    return max(1, min(kRebuildBlocks, most));
}

void launch_cells(const Bufs& b, int precision, int ntiles, int nsys, int force_all,
                  cudaStream_t s, long* launches) {
    if (ntiles <= 0) return;
    if (b.rtiles) launch_next(k_rebuild_list, 1, 256, s, b, nsys, force_all);
    const int g = rebuild_grid(b, ntiles);
    if (precision == NEFE_FP64) launch_next(k_cells_count<double>, g, kTile, s, b);
    else launch_next(k_cells_count<float>, g, kTile, s, b);
    if (!b.rtiles && b.scan_sums && b.ncells_host > kScanOneBlock) {
        const int span = cells_scan_span(b.ncells_host);
        const int blocks = (b.ncells_host + span - 1) / span;
        launch_next(k_cells_span_sums, blocks, 256, s, b, span, b.scan_sums);
        launch_next(k_cells_scan_spans, blocks, 256, s, b, span, b.scan_sums);
    } else {
        launch_next(k_cells_scan, nsys, 256, s, b, force_all || !b.rtiles);
    }
    if (precision == NEFE_FP64) launch_next(k_cells_fill<double>, g, kTile, s, b);
    else launch_next(k_cells_fill<float>, g, kTile, s, b);
    if (launches) *launches += 4;
}

int cells_scan_span(int ncells) {
    const int per = (ncells + kScanBlocks - 1) / kScanBlocks;
    return (per + 2047) / 2048 * 2048;
}

void launch_cells_sort(const Bufs& b, int ncells, cudaStream_t s) {
    const int blocks = (ncells + 255) / 256;
    launch_next(k_cells_sort, blocks < 4096 ? blocks : 4096, 256, s, b);
}

int cells_by_flag(int nsys, int ntiles) { return nsys <= kClusterSystems && ntiles <= kClusterTiles ? 1 : 0; }

void launch_cells_and_list(const Bufs& b0, int precision, int ntiles, int nsys, int force_all,
                           cudaStream_t s, long* launches) {
    Bufs b = b0;
    if (force_all || b.list_lanes != 0) b.by_flag = 0;   // (the worklist's own kernels)
    if (ntiles <= 0) return;
    if (force_all || !b.by_flag) {
        launch_cells(b, precision, ntiles, nsys, force_all, s, launches);
    } else {
        if (precision == NEFE_FP64) launch_next(k_cells_clusters<double>, nsys * kCellsCluster, kCellsThreads, s, b, nsys);
        else launch_next(k_cells_clusters<float>, nsys * kCellsCluster, kCellsThreads, s, b, nsys);
        if (launches) *launches += 1;
    }
    const int L = (b.list_lanes == 8 || b.list_lanes == 16 || b.list_lanes == 32) ? b.list_lanes : 0;
    if (L == 0) {
        const int g = list_grid(b, ntiles);
        if (precision == NEFE_FP64) launch_next(k_nlist_cell<double>, g, kTile, s, b, nsys);
        else launch_next(k_nlist_cell<float>, g, kTile, s, b, nsys);
        if (launches) *launches += 1;
        return;
    }
    const int g = rebuild_grid(b, ntiles * L);
    if (precision == NEFE_FP64) {
        if (L == 8) launch_next(k_nlist<double, 8>, g, kTile, s, b);
        else if (L == 16) launch_next(k_nlist<double, 16>, g, kTile, s, b);
        else launch_next(k_nlist<double, 32>, g, kTile, s, b);
    } else {
        if (L == 8) launch_next(k_nlist<float, 8>, g, kTile, s, b);
        else if (L == 16) launch_next(k_nlist<float, 16>, g, kTile, s, b);
        else launch_next(k_nlist<float, 32>, g, kTile, s, b);
    }
    if (launches) *launches += 1;
}

int rebuild_coop_blocks(int precision) {
    int per_sm = 0, dev = 0, sms = 0;
    cudaError_t e = precision == NEFE_FP64
                        ? cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_rebuild_coop<double>, kTile, 0)
                        : cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_rebuild_coop<float>, kTile, 0);
    if (e != cudaSuccess || cudaGetDevice(&dev) != cudaSuccess ||
        cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return min(per_sm * sms, kRebuildBlocks);
}

void launch_rebuild_coop(const Bufs& b0, int precision, int blocks, int nsys, cudaStream_t s, long* launches) {
    Bufs b = b0;
    b.by_flag = 0;                               // (its own worklist)
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = dim3((unsigned)blocks);
    cfg.blockDim = dim3(kTile);
    cfg.dynamicSmemBytes = 0;
    cfg.stream = s;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeCooperative;   // every block resident: the grid barriers can complete
    at[0].val.cooperative = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    if (precision == NEFE_FP64) cudaLaunchKernelEx(&cfg, k_rebuild_coop<double>, b, nsys);
    else cudaLaunchKernelEx(&cfg, k_rebuild_coop<float>, b, nsys);
    if (launches) *launches += 1;
}

int check_barrier_timeout(double limit_ms) {
    void* p = nullptr;
    if (cudaMalloc(&p, 2 * sizeof(int)) != cudaSuccess) return -2;
    cudaMemset(p, 0, 2 * sizeof(int));
    unsigned* word = static_cast<unsigned*>(p);
    int* tmo = static_cast<int*>(p) + 1;
    k_barrier_selftest<<<4, kTile>>>(word, tmo, (unsigned long long)(limit_ms * 1e6));
    int h = 0;
    const cudaError_t e = cudaMemcpy(&h, tmo, sizeof(int), cudaMemcpyDeviceToHost);
    cudaFree(p);
    if (e != cudaSuccess) return -3;
    return h ? 1 : 0;
}

void launch_aos_soa(const double* src, double* dst, int n, int to_soa, cudaStream_t s) {
    if (n <= 0) return;
    const int blocks = (3 * n + 255) / 256;
    if (to_soa) launch_next(k_aos_to_soa, blocks, 256, s, src, dst, n);
    else launch_next(k_soa_to_aos, blocks, 256, s, src, dst, n);
}

__global__ void k_decode_grad(const long long* acc, double* out8) {
    dep_wait();
    const int t = threadIdx.x;
    if (t >= 8) return;
    const int a = t == 0 ? ACC_UINT : ACC_DTH + (t - 1);
    out8[t] = decoded(acc, a);
}

void launch_decode_grad(const long long* acc, double* out8, cudaStream_t s) {
    launch_next(k_decode_grad, 1, 32, s, acc, out8);
}

void launch_decode_ev(const long long* acc, double* out7, const unsigned* err, cudaStream_t s) {
    launch_next(k_decode_ev, 1, 32, s, acc, out7, err);
}

void launch_uf_list(const Bufs& b0, int precision, int ntiles, int nsys, int force_all, cudaStream_t s, long* launches) {
    Bufs b = b0;
    if (force_all || b.list_lanes != 0) b.by_flag = 0;
    if (ntiles <= 0 || !b.uf_nbr) return;
    const int g = list_grid(b, ntiles);
    if (precision == NEFE_FP64) launch_next(k_uflist<double>, g, kTile, s, b, nsys);
    else launch_next(k_uflist<float>, g, kTile, s, b, nsys);
    if (launches) *launches += 1;
}

void launch_uf(const Bufs& b, int precision, int ntiles, int mode, cudaStream_t s, long* launches) {
    if (ntiles <= 0 || !b.uf_nbr) return;
    if (precision == NEFE_FP64) {
        if (mode == FM_FORCES) launch_next(k_uf<double, FM_FORCES, false>, ntiles * kUfBlocks<double>, kUfThreads<double>, s, b);
        else launch_next(k_uf<double, FM_STEP, false>, ntiles * kUfBlocks<double>, kUfThreads<double>, s, b);
    } else {
        const auto go = [&](auto kernel) { launch_next(kernel, ntiles * kUfBlocks<float>, kUfThreads<float>, s, b); };
        if (mode == FM_FORCES) b.want_xf > 1 ? go(k_uf<float, FM_FORCES, true>) : go(k_uf<float, FM_FORCES, false>);
        else b.want_xf > 1 ? go(k_uf<float, FM_STEP, true>) : go(k_uf<float, FM_STEP, false>);
    }
    if (launches) *launches += 1;
}

void launch_kick_drift(const Bufs& b, int precision, int ntiles, int mode, cudaStream_t s, long* launches,
                       int skip, int drawn) {
    if (ntiles <= 0) return;
    if (precision == NEFE_FP64) launch_next(k_kick_drift<double>, ntiles, kTile, s, b, mode, skip, drawn);
    else launch_next(k_kick_drift<float>, ntiles, kTile, s, b, mode, skip, 0);
    if (launches) *launches += 1;
}

void launch_positions(const Bufs& b, int precision, int ntiles, cudaStream_t s, long* launches) {
    if (ntiles <= 0) return;
    if (precision == NEFE_FP64) launch_next(k_positions<double>, ntiles, kTile, s, b);
    else launch_next(k_positions<float>, ntiles, kTile, s, b);
    if (launches) *launches += 1;
}

// Fractional positions only (stateless scatter form).
__global__ void __launch_bounds__(kTile) k_frac_positions(Bufs b) {
    dep_wait();
    const int i = blockIdx.x * kTile + threadIdx.x;
    if (i >= b.ntot) return;
    const size_t N = b.ntot;
    const double x[3] = {b.x[i], b.x[N + i], b.x[2 * N + i]};
    const int4 f = frac_position(x, b.st[0], b.want_xf > 1);
    b.xf[i] = f;
    b.xc[i] = pack_frac(f);
    if (i == 0) scale_of_box(b, 0, b.st[0]);
}
void launch_frac_positions(const Bufs& b, cudaStream_t s) {
    if (b.ntot > 0) launch_next(k_frac_positions, (b.ntot + kTile - 1) / kTile, kTile, s, b);
}

void launch_mirror(const Bufs& b, int precision, int ntiles, cudaStream_t s, long* launches) {
    if (ntiles <= 0) return;
    if (precision == NEFE_FP64) launch_next(k_mirror<double>, ntiles, kTile, s, b);
    else launch_next(k_mirror<float>, ntiles, kTile, s, b);
    if (launches) *launches += 1;
}

// Atoms per warp of the edge-list kernels, as a power of two: by the whole context's size, so that a
// run does not depend on how the passes are launched.  FP32 (see k_edges_s): 32 where that gives every
// SM 8 warps, else 16 or 8.  FP64, where one warp a SM quarter fills the unit: 16 (32 atoms' edges do
// not fit one list) where that gives 4 warps a SM, 8 down to 2 warps, else 4.
int atoms_per_warp_log2(int precision, int ntot) {
    if (precision == NEFE_FP64) return ntot >= 16 * 152 * 4 ? 4 : ntot >= 8 * 152 * 2 ? 3 : 2;
    return ntot >= 32 * 152 * 8 ? 5 : ntot >= 16 * 152 * 8 ? 4 : 3;
}

// The last quarter of what the chip holds at once is cut into blocks of half the size, where there is
// more than that to do: the launch ends on the SMs that drew the last blocks.  Pass A without and with
// it: liquid, 192,000 atoms 77.4 -> 74.6 us, 256,000 88.5 -> 86.6, 1,024,000 313.5 -> 309.9; beta-tin 176,000
// 79.4 -> 76.6, 512,000 179.5 -> 175.3; crystal (skin 1.6 A) 192,000 36.9 -> 36.1, 1,024,000 152.2 -> 151.3; FP64
// crystal 48,000 158.8 -> 154.6, 128,000 355.6 -> 352.1.  It costs crystals whose last filling is between three
// quarters and full anyway: 256,000 atoms 38.9 -> 41.1 us, 384,000 55.8 -> 58.2 (liquids and beta-tin gain 2 %
// there).  A larger share or quarter-size blocks give less, their lists being shorter, and just above one
// filling (136,000 atoms) it costs 5 %.
void set_edge_items(Bufs& b, int precision, int lg, int ntiles) {
    const int resident = 152 * (precision == NEFE_FP64 ? kEdgesDBlocks : kScatterBlocks);
    const bool cut = (long long)ntiles << (6 - lg) > resident + resident / 4;
    b.lg = lg;
    b.lg_tail = max(2, lg - 1);
    b.tail_tile = cut ? ntiles - (resident / 4 >> (6 - lg)) : ntiles;
}
static int edge_items(const Bufs& b, int ntiles) {
    const int big = max(0, min(b.tail_tile - b.tile_base, ntiles));
    return (big << (6 - b.lg)) + ((ntiles - big) << (6 - b.lg_tail));
}

static void edges_fp32(const Bufs& b, int lanes, int ntiles, cudaStream_t s) {
    switch (lanes) {
        case 0: {
            const int items = edge_items(b, ntiles);
            const auto go = [&](auto kernel) { launch_next_if(!b.uf_nbr || items <= kEarlyBlocks, kernel, items, kScatterThreads, s, b, b.swc_common); };
            const bool full = items >= 152 * kScatterBlocks;
            if (b.want_xf > 1) {
                if (b.want_grad) go(k_edges_s<false, true, true, kScatterBlocks, true>);
                else if (b.e_atom) go(k_edges_s<true, false, true, kScatterBlocks, true>);
                else if (!b.common) go(k_edges_s<false, false, false, kScatterBlocks, true>);
                else go(k_edges_s<false, false, true, kScatterBlocks, true>);
            } else if (b.want_grad) go(k_edges_s<false, true, true, kScatterBlocks, false>);   // (stateless: one system)
            else if (b.e_atom) go(k_edges_s<true, false, true, kScatterBlocks, false>);
            else if (!b.common) go(k_edges_s<false, false, false, kScatterBlocks, false>);
            else if (full) go(k_edges_s<false, false, true, kScatterBlocks, false>);
            else go(k_edges_s<false, false, true, kScatterBlocksFew, false>);
            break;
        }
        case 1: launch_next(k_edges1<float>, ntiles * (kTile / kEdges1Threads), kEdges1Threads, s, b); break;
        case 4: launch_next(k_edges<float, 4>, ntiles * 4, kTile, s, b); break;
        case 8: launch_next(k_edges<float, 8>, ntiles * 8, kTile, s, b); break;
        case 16: launch_next(k_edges<float, 16>, ntiles * 16, kTile, s, b); break;
        default: launch_next(k_edges<float, 32>, ntiles * 32, kTile, s, b); break;
    }
}

static void edges_fp64(const Bufs& b, int ntiles, cudaStream_t s) {
    const int items = edge_items(b, ntiles);
    Bufs bn = b;
    bn.noise_first = b.noise_ahead ? items : -1;
    const int blocks = items + (b.noise_ahead ? 4 * ntiles : 0);
    const auto go = [&](auto kernel) { launch_next_if(!b.uf_nbr || blocks <= kEarlyBlocks, kernel, blocks, 64, s, bn, b.swp_common); };
    if (b.want_grad) go(k_edges_d<true, true>);          // (stateless: one system)
    else if (b.common) go(k_edges_d<false, true>);
    else go(k_edges_d<false, false>);
}

void launch_edges(const Bufs& b, int precision, int lanes, int ntiles, int mode, cudaStream_t s,
                  long* launches) {
    (void)mode;
    if (ntiles <= 0) return;
    if (precision == NEFE_FP64) edges_fp64(b, ntiles, s);
    else edges_fp32(b, lanes, ntiles, s);
    if (launches) *launches += 1;
}

template <typename T, int MODE>
static void gather_dispatch(const Bufs& b, int lanes, int ntiles, cudaStream_t s, int fuse) {
    switch (lanes) {
        case 0: launch_next_if(ntiles <= kEarlyBlocks, k_finish<T, MODE>, ntiles, kTile, s, b, fuse); break;
        case 1: launch_next_if(ntiles <= kEarlyBlocks, k_gather<T, MODE, 1>, ntiles, kTile, s, b); break;
        case 2: launch_next_if(ntiles * 2 <= kEarlyBlocks, k_gather<T, MODE, 2>, ntiles * 2, kTile, s, b); break;
        case 8: launch_next_if(ntiles * 8 <= kEarlyBlocks, k_gather<T, MODE, 8>, ntiles * 8, kTile, s, b); break;
        default: launch_next_if(ntiles * 4 <= kEarlyBlocks, k_gather<T, MODE, 4>, ntiles * 4, kTile, s, b); break;
    }
}

void launch_gather(const Bufs& b, int precision, int lanes, int ntiles, int mode, cudaStream_t s,
                   long* launches, int fuse) {
    if (ntiles <= 0) return;
    if (precision == NEFE_FP64) {
        if (mode == FM_FORCES) gather_dispatch<double, FM_FORCES>(b, lanes, ntiles, s, 0);
        else if (mode == FM_SETUP) gather_dispatch<double, FM_SETUP>(b, lanes, ntiles, s, 0);
        else gather_dispatch<double, FM_STEP>(b, lanes, ntiles, s, fuse);
    } else {
        if (mode == FM_FORCES) gather_dispatch<float, FM_FORCES>(b, lanes, ntiles, s, 0);
        else if (mode == FM_SETUP) gather_dispatch<float, FM_SETUP>(b, lanes, ntiles, s, 0);
        else gather_dispatch<float, FM_STEP>(b, lanes, ntiles, s, fuse);
    }
    if (launches) *launches += 1;
}

void launch_materialize(const Bufs& b, int precision, int ntiles, double* x, double* v, cudaStream_t s) {
    if (ntiles <= 0) return;
    if (precision == NEFE_FP64) launch_next(k_materialize<double>, ntiles, kTile, s, b, x, v);
    else launch_next(k_materialize<float>, ntiles, kTile, s, b, x, v);
}

void launch_inject(const Bufs& b, int precision, int ntiles, const double* x, const double* v, cudaStream_t s) {
    if (ntiles <= 0) return;
    if (precision == NEFE_FP64) launch_next(k_inject<double>, ntiles, kTile, s, b, x, v);
    else launch_next(k_inject<float>, ntiles, kTile, s, b, x, v);
}

void launch_group(const Bufs& b, const DevGroup* groups, int ngroups, int mode, cudaStream_t s,
                  long* launches, int carry) {
    if (ngroups <= 0) return;
    launch_next_if(ngroups <= kEarlyGroups, k_group, ngroups, kTile, s, b, groups, mode, carry);
    if (launches) *launches += 1;
}

void launch_noise(unsigned long long seed, unsigned long long sys_id, unsigned long long step, int n,
                  int precision, double* xi, cudaStream_t s) {
    if (n <= 0) return;
    launch_next(k_noise, (n + 127) / 128, 128, s, seed, sys_id, step, n, precision, xi);
}

}  // namespace nefe
