// Host-side launchers of the libnefe kernels (defined in nefe_kernels.cu).
#pragma once
#include <cuda_runtime.h>
#include "nefe_dev.h"
#include "nefe_sw_terms.h"

namespace nefe {

constexpr int kSlots = 32;   // accumulator slots per system (spreads atomics over 32 words)

// Pointers handed to every kernel.  Per-atom arrays are global over all systems of a
// context; FP64 SoA arrays have stride ntot.  F/xs/xsb are float4 (FP32 path) or double4.
struct Bufs {
    const DevSys* sys;
    DevState* st;
    long long* acc;          // [nsys][ACC_N][kSlots]
    long long* acc_lo;       // remainders of the sums in 2^-40 units: stateless, an array of the same layout;
                             // FP64 engine, acc itself (engine_lo_row); or NULL
    const int4* tiles;       // 128-atom tiles: system, first atom, atom count
    double* x;               // FP64 anchor positions (positions at the last list build), SoA
    void* dhi;               // displacement since the last build, kernel precision, SoA (may be NULL)
    void* dlo;               // its compensation term (FP32 path; may be NULL)
    void* v;                 // velocities, kernel precision, SoA
    const double* r0;        // Einstein sites, FP64 SoA
    void* F;                 // total force used by the next half kick (T4)
    void* xs;                // mirror x - q h (T4)
    void* xa;                // mirror at the last build (T4)
    void* xcs;               // mirror at the last build in cell order, atom index in .w (T4)
    void* sd0;               // anchor - r0 at the last build (T4)
    void* xi;                // thermostat noise of the current step (T4)
    void* shd;               // [ntot][kShell] in-cutoff shell: d_ij and g_ij (T4)
    int* shj;                // [ntot][kShell] shell neighbour indices
    int* shn;                // shell size (FP64: entries, and << 16 those of them outside the cutoff)
    void* spill;             // thread-per-atom pass A: shell entries beyond its shared table, or NULL
    void* P;                 // [ntot] pass-A force (.w = atom energy), then in FP32 [ntot][2] its virial (T4)
    int4* q;                 // unwrapped cell index per axis, from the last build
    int* cell_of;
    int* perm;
    int* cell_start;         // per system: ncell_cap + 1 entries at cell0 + system index
    int* cell_count;
    int* cell_cursor;
    int* nbr;
    int* cnt;
    int cap;
    int nbr_il;              // 0: rows row-major (entry k of atom i at i cap + k); 1 (engine, cap a
                             // multiple of 4): interleaved by 4 -- entries 4g..4g+3 of every atom
                             // form one 16-byte vector, the vectors of consecutive atoms adjacent
                             // (at (g ntot + i) 4 + k % 4), and each row is padded to a multiple
                             // of 4 with entries that never pass the distance test
    int ntot;
    int tile_base;           // first tile of the launch (force passes run in L2-sized chunks)
    int* rtiles;             // rebuild worklist (tiles of flagged systems) or NULL
    int* rcount;             // its length
    int* rcbase;             // [nsys + 1] first worklist cell of each system (cells of flagged
                             // systems, in system order; the last entry is their number) or NULL
    double dt;
    const void* swc;         // SWc<float> (FP32) or SWp<double> (FP64) table
    DevPair* pairs;
    double* trace;
    double* f_out;           // stateless: FP64 SoA forces
    double* e_atom;          // stateless: per-atom energy (may be NULL)
    int want_grad;           // pass A also sums dE/d(A, B, p, q, a, lambda3, gamma)
    int list_lanes;          // list build: 0 one warp per cell; 8, 16 or 32 lanes per atom
    int* uf_nbr;             // [ntot][kUfCap] Uhlenbeck-Ford pair rows (NULL: no UF system)
    int* uf_cnt;             // [ntot] their lengths
    void* uf_F;              // [ntot] UF force and atom energy of the step (T4)
    const int* uf_tiles;     // tiles of the UF systems (per-step UF kernel), or NULL: every tile
    int* scan_sums;          // stateless: span sums of a multi-block cell scan (NULL: one block)
    int by_flag;             // small context: cells by k_cells_clusters, list builds by the rebuild flags
    int ncells_host;         // number of cells of the grid (engine: of all systems at creation)
    int* lacc;               // [ntot][4] int32 force accumulators of the scatter form (2^-22 eV/A)
    long long* lacc_hi;      // [ntot][3] multiples of large terms (see k_edges_s)
    SWc<float> swc_common;   // the potential constants, where every system has the same (common)
    SWp<double> swp_common;
    int lg;                  // atoms per warp of the edge-list kernels, as a power of two
    void* xi_next;           // FP64: noise drawn ahead by pass A (noise_ahead), 4 doubles per atom, or NULL
    int noise_ahead, noise_first;   // draw it in this launch; first block that does (-1: none)
    int lg_tail, tail_tile;  // the same from tile tail_tile on (set_edge_items)
    int common;
    int leg_refuse;          // the scatter form was chosen by the caller: terms above its limit are refused
    int* hi_flag;            // [tiles] some large term was split this step (cleared by k_finish)
    float4* lscale;          // [nsys][4] L 2^-32 as FP32 value and remainder, 1 - h/hb, 2^32/L
    int4* xf;                // FP32: fractional positions (x/L as 32-bit fixed point)
    int4* xfb;               // their values at the last list build
    uint2* xc;               // their top 21 bits per axis (pass A's row filter)
    int want_xf, want_xs;    // per-step positions: fractional (scatter form; FP64: xc only; 2: with ten more
                             // bits an axis in .w, see kFracCoarse), FP32 mirror (the others)
    int row4;                // row-major rows can be read 16 bytes at a time
    int* any_rebuild;        // engine: [0] some system's rebuild flag is set this step, [1] some
                             // rebuild_next is set (fused epilogue); NULL in the stateless calls
    int rebuild_all;         // engine: when any system's list is stale, every system rebuilds (one
                             // full-width build instead of many narrow ones)
};

enum ForceMode { FM_FORCES = 0, FM_SETUP = 1, FM_STEP = 2 };

// Cell count / scan / fill only.
void launch_cells(const Bufs& b, int precision, int ntiles, int nsys, int force_all,
                  cudaStream_t s, long* launches);
// Orders the atoms of each cell by index (the stateless cell sort, after launch_cells).
void launch_cells_sort(const Bufs& b, int ncells, cudaStream_t s);
// Cells per block of the multi-block scan (its scratch: one int per block, at most 1024).
int cells_scan_span(int ncells);
// Decodes one system's fixed-point sums into [U_int, virial xx yy zz xy xz yz] (FP64, device); NaN
// where the error word says that a block's sum is missing (err: device, or NULL).
void launch_decode_ev(const long long* acc, double* out7, const unsigned* err, cudaStream_t s);
// Decodes [U_int, dE/dA, dE/dB, dE/dp, dE/dq, dE/da, dE/dlambda3, dE/dgamma] (FP64, device).
void launch_decode_grad(const long long* acc, double* out8, cudaStream_t s);
// Rebuild sequence (only systems whose rebuild flag is set, or all when force_all).
void launch_cells_and_list(const Bufs& b, int precision, int ntiles, int nsys, int force_all,
                           cudaStream_t s, long* launches);
// Half kick + drift + mirror + displacement check + noise sums (mode 0: no kick/drift).  skip:
// the systems without a barostat were moved by the previous step's fused epilogue.
void launch_kick_drift(const Bufs& b, int precision, int ntiles, int mode, cudaStream_t s,
                       long* launches, int skip = 0, int drawn = 0);
// Uhlenbeck-Ford pair rows of the UF systems (after the cell fill; flagged systems only when a
// rebuild worklist is set).
void launch_uf_list(const Bufs& b, int precision, int ntiles, int nsys, int force_all, cudaStream_t s, long* launches);
// Uhlenbeck-Ford forces and energies over `ntiles` tiles (b.uf_tiles, or every tile when NULL);
// mode FM_FORCES writes b.f_out / b.e_atom (stateless), otherwise b.uf_F for pass B.
void launch_uf(const Bufs& b, int precision, int ntiles, int mode, cudaStream_t s, long* launches);
int cells_by_flag(int nsys, int ntiles);   // value of by_flag for a context
int atoms_per_warp_log2(int precision, int ntot);
void set_edge_items(Bufs& b, int precision, int lg, int ntiles);
// Force pass A (edges: pair terms, triplets centred on each atom, leg forces per edge).
void launch_edges(const Bufs& b, int precision, int lanes, int ntiles, int mode, cudaStream_t s,
                  long* launches);
// Force pass B (gather leg forces; springs, Langevin and second half kick in FM_SETUP/FM_STEP).
// fuse (scatter form, FM_STEP): systems without a barostat go on to the next step's kick, drift
// and noise in the same kernel.
void launch_gather(const Bufs& b, int precision, int lanes, int ntiles, int mode, cudaStream_t s,
                   long* launches, int fuse = 0);
// FP64 positions (anchor + displacement) and FP64 velocities into SoA staging buffers.
void launch_materialize(const Bufs& b, int precision, int ntiles, double* x, double* v, cudaStream_t s);
// Replace positions (anchor, zero displacement) and/or velocities from FP64 SoA buffers.
void launch_inject(const Bufs& b, int precision, int ntiles, const double* x, const double* v, cudaStream_t s);
// Per-group scalar update. mode 0 INIT, 1 STEP, 2 OBSERVE.  carry (STEP): the previous epilogue
// was fused (its next-step noise sums and rebuild flag are moved into place).
void launch_group(const Bufs& b, const DevGroup* groups, int ngroups, int mode, cudaStream_t s,
                  long* launches, int carry = 0);
// Positions of every atom from anchor and displacement, in the forms in use (want_xf, want_xs).
void launch_positions(const Bufs& b, int precision, int ntiles, cudaStream_t s, long* launches);
// Fractional positions of b.x (stateless scatter form).
void launch_frac_positions(const Bufs& b, cudaStream_t s);
// Mirror only (stateless force entry): q and xs from x with the list-build formula.
void launch_mirror(const Bufs& b, int precision, int ntiles, cudaStream_t s, long* launches);
// Thermostat noise as FP64 (n,3).
void launch_noise(unsigned long long seed, unsigned long long sys_id, unsigned long long step,
                  int n, int precision, double* xi, cudaStream_t s);

// The engine's single-launch rebuild (cooperative; see k_rebuild_coop): the largest grid whose
// blocks are all resident (0 if it cannot be launched), and its launch.
int rebuild_coop_blocks(int precision);
void launch_rebuild_coop(const Bufs& b, int precision, int blocks, int nsys, cudaStream_t s, long* launches);
// Runs the barrier time-limit check on the current device: 1 timed out (expected), 0 did not,
// negative on a CUDA error.
int check_barrier_timeout(double limit_ms);

bool lanes_supported(int lanes);
// (n,3) row-major <-> SoA (to_soa = 1: aos -> soa).
void launch_aos_soa(const double* src, double* dst, int n, int to_soa, cudaStream_t s);

}  // namespace nefe
