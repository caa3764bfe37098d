// Device code of the DI-LBM step on sm_103a.
//
// One time step (the paper's procedure, Sec. 2.3) is two kinds of work, which
// run side by side in one launch over many steps (run_steps):
//   the sweep     -- every node: pull-stream, edge extrapolation, solid
//                    fraction (Eq. 14), corrected velocity (Eq. 17),
//                    collision with the force term (Eqs. 13, 15), and the
//                    node's share of force/torque (Eqs. 18-19) summed per
//                    row segment and nearby particle;
//   the particles -- one warp per particle: Wan-Turek repulsion (Eqs. 28-29),
//                    fixed-order FP64 sum of its partials (Eqs. 18-19) once
//                    they are all there, Newton-Euler update (Eqs. 22-24),
//                    then binning of the particle into the lattice tiles its
//                    phi tail reaches, for the next sweep.
//
// Populations are stored as deviations d_i = f_i - w_i (a context's row by row:
// the nine directions' rows of `pitch` elements one after another, so that a
// sweep moves through one stretch of memory and not through nine at once), in
// FP32, FP16 or BF16; arithmetic
// is FP32, force/torque accumulation and particle state FP64.  Particle
// positions and the tile bins are double-buffered by step parity, so a step
// reads one copy and writes the other.
//
// The sweep is persistent: each warp takes row segments of 128 nodes
// and streams every segment's nine source rows (plus a 16-byte halo on each
// side) into shared memory with bulk asynchronous copies (cp.async.bulk,
// completion on an mbarrier); once a segment's rows have been read, the copy
// of the warp's next segment is issued into the same buffer, so it is in
// flight while the current segment is collided.  Each lane sweeps its four
// nodes as two pairs (nodes 2l, 2l + 1 of each half segment), which keeps
// few registers live; writes go straight from registers, one contiguous run
// per plane and pair.
//
// Two launches a step (sweep, particles) against this, us per step (FP32 unless
// said, default shapes): 200 x 100 cylinder 18.5 -> 8.0, 400 x 2000 box
// 36.9 -> 15.9, 1793 x 179 channel in FP16 21.6 -> 11.7, 512^2 suspension
// 22.6 -> 11.5, 501 x 101 channel with a moving frame 30.8 -> 8.8, 64 uneven
// lattices 264 -> 231, 4096^2 suspension 225.6 -> 211 (FP16 221.4 -> 198, PS
// 247 -> 228).
#pragma once

#include <cuda_bf16.h>
#include <type_traits>
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

namespace dilbm {

constexpr int TILE_W = 128;   // nodes per row segment (32 lanes x 4 nodes) and per tile row
constexpr int TILE_H = 8;     // rows per binning tile
constexpr int TILE_W_LOG2 = 7, TILE_H_LOG2 = 3;
static_assert(TILE_W == 1 << TILE_W_LOG2 && TILE_H == 1 << TILE_H_LOG2, "tiles of a power of two");
constexpr int MAXC = 32;      // candidate particles per tile
constexpr int MAXT = 128;     // tiles one particle's phi tail may reach
constexpr int NREC = 3;       // float4 records per binned particle
constexpr int SWEEP_WARPS = 8;   // default row segments in flight per block of the sweep alone (one per warp)
constexpr int GUARD = 256;    // elements kept readable before and after a population buffer
constexpr float PHI_CUT_WIDTHS = 4.0f;   // phi tail kept up to 4 interface widths (phi > 1.1e-7)
constexpr unsigned long long WAIT_LIMIT_NS = 1000000000ull;   // bounded device waits: 1 s

enum : int { SIDE_PERIODIC = 0, SIDE_VELOCITY = 1, SIDE_PRESSURE = 2,
             SIDE_HALO = 3 };   // a strip's cut: the rows beyond it come from halo buffers
enum : int { WEST = 0, EAST = 1, SOUTH = 2, NORTH = 3 };
enum : int { ERR_UNSTABLE = 1, ERR_OVERFLOW = 2, ERR_TIMEOUT = 4, ERR_BADPARTICLE = 8 };

// D2Q9 directions of Eq. 3 and weights of Eq. 4.
__host__ __device__ constexpr int cxof(int i) { return i == 1 || i == 5 || i == 8 ? 1 : (i == 3 || i == 6 || i == 7 ? -1 : 0); }
__host__ __device__ constexpr int cyof(int i) { return i == 2 || i == 5 || i == 6 ? 1 : (i == 4 || i == 7 || i == 8 ? -1 : 0); }
__host__ __device__ constexpr float wof(int i) { return i == 0 ? 4.0f / 9.0f : (i <= 4 ? 1.0f / 9.0f : 1.0f / 36.0f); }

// ------------------------------------------------------------ storage types
template <typename T> struct Storage;

template <> struct Storage<float> {
    static __device__ __forceinline__ float load1(const float *p) { return __ldcg(p); }
    static __device__ __forceinline__ float lds1(const float *p) { return *p; }
    static __device__ __forceinline__ void store1(float *p, float v) { *p = v; }
    static __device__ __forceinline__ float2 lds2(const float *p) { return *reinterpret_cast<const float2 *>(p); }
    static __device__ __forceinline__ void store2(float *p, float2 v) { *reinterpret_cast<float2 *>(p) = v; }
};

template <> struct Storage<__half> {
    static __device__ __forceinline__ float load1(const __half *p) { return __half2float(__ldcg(p)); }
    static __device__ __forceinline__ float lds1(const __half *p) { return __half2float(*p); }
    static __device__ __forceinline__ void store1(__half *p, float v) { *p = __float2half_rn(v); }
    static __device__ __forceinline__ float2 lds2(const __half *p) { return __half22float2(*reinterpret_cast<const __half2 *>(p)); }
    static __device__ __forceinline__ void store2(__half *p, float2 v) { *reinterpret_cast<__half2 *>(p) = __floats2half2_rn(v.x, v.y); }
};

template <> struct Storage<__nv_bfloat16> {
    static __device__ __forceinline__ float load1(const __nv_bfloat16 *p) { return __bfloat162float(__ldcg(p)); }
    static __device__ __forceinline__ float lds1(const __nv_bfloat16 *p) { return __bfloat162float(*p); }
    static __device__ __forceinline__ void store1(__nv_bfloat16 *p, float v) { *p = __float2bfloat16_rn(v); }
    static __device__ __forceinline__ float2 lds2(const __nv_bfloat16 *p) {
        return __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(p));
    }
    static __device__ __forceinline__ void store2(__nv_bfloat16 *p, float2 v) {
        *reinterpret_cast<__nv_bfloat162 *>(p) = __floats2bfloat162_rn(v.x, v.y);
    }
};

// Elements in the 16-byte halo on each side of a staged row segment, and the
// staged width.
template <typename T> __host__ __device__ constexpr int halo_of() { return 16 / (int)sizeof(T); }
template <typename T> __host__ __device__ constexpr int segw_of() { return TILE_W + 2 * halo_of<T>(); }

// Elements of one stage: the 9 staged rows.
template <typename T> __host__ __device__ constexpr int stage_elems() { return 9 * segw_of<T>(); }

// Dynamic shared memory of one sweep block of W warps.
template <typename T, int W = SWEEP_WARPS> __host__ __device__ constexpr size_t sweep_smem_bytes() {
    return (size_t)W * stage_elems<T>() * sizeof(T)             // staged rows
           + (size_t)W * MAXC * (NREC + 1) * sizeof(float4)     // candidate records and force sums
           + (size_t)W * MAXC * sizeof(int)                     // candidate ids
           + (size_t)W * sizeof(uint64_t);                      // mbarriers
}

// ------------------------------------------------------------ parameters
struct Particles {      // structure of arrays, device memory
    double *x[2], *y[2];        // centre, by step parity
    float *xf[2], *yf[2];       // FP32 copy of the centre, for cheap proximity tests
    double *r, *ux, *uy, *omega, *theta, *rho_s;
    // formed when the particles are uploaded: 1 / m and 1 / I (Eqs. 22-23), the
    // buoyancy-reduced weight in x and y, and the reach (r + the phi tail)
    double *im, *iI, *wx, *wy, *reach;
    float *rf;                  // r in FP32
    int *fixed;
};

struct Lattice {
    int nx, ny, pitch;          // nodes; row pitch in elements (multiple of 32)
    // Elements from a direction's row to the next direction's and from a row to
    // the next: pitch and 9 * pitch in a context, ny * pitch and pitch in the
    // static step's planes (its caller's layout).  Rows against planes on 4096^2,
    // us per step less: FP32 1.3, FP16 2.1, PS 2.2.
    long long plane, row;
    int ntx, nty;               // tiles along x and y
    bool per_x, per_y;          // periodic axes
    bool wrap_x, wrap_y;        // periodic and short enough that a tile's nodes
                                // need their own minimum image
    int side_kind[4];
    float side_ux[4], side_uy[4], side_drho[4];   // drho = rho_b - 1
    // 16-bit storage holds s_i = (d_i - e_i) / q: d_i = f_i - w_i the FP32
    // deviation, e_i the deviation of the lattice's initial equilibrium
    // f^eq(rho_init, u0) and q a power of two that keeps small s_i out of
    // the FP16 subnormals.  FP32 storage holds d_i itself.
    float ref_e[9];             // e_i
    float ref_q, ref_iq;        // q, 1 / q
    // The moments of the reference e_i (it is the equilibrium deviation of
    // Eq. 2 at rho_init, u0): m0 = rho_init - 1, B = rho_init u0,
    // M = rho_init u0 u0^T (xx, yy, xy), in the moment form below.  The
    // 16-bit sweep takes moments of the stored s_i and adds these, so no
    // per-direction offset enters its inner loop.
    float ref_m[6];
    // A strip of a larger lattice (one rank's rows): the post-collision rows
    // just south (halo[0]) and north (halo[1]) of it, 9 plane rows of `pitch`
    // elements each, with GUARD readable elements before and after; NULL
    // where the side is a physical side of the lattice.
    const void *halo[2];
};

// Is row y of the lattice a south / north edge row (a physical side, not a
// periodic axis and not a strip's cut)?
__host__ __device__ inline bool south_edge_row(const Lattice &L, int y) {
    return !L.per_y && y == 0 && L.side_kind[SOUTH] != SIDE_HALO;
}
__host__ __device__ inline bool north_edge_row(const Lattice &L, int y) {
    return !L.per_y && y == L.ny - 1 && L.side_kind[NORTH] != SIDE_HALO;
}

// Stored value <-> FP32 deviation d_i for direction i (exact scalings by a
// power of two, one rounding in the offset).
template <typename T> __device__ __forceinline__ float from_store(const Lattice &L, int i, float v) {
    if constexpr (std::is_same<T, float>::value) return v;
    else return fmaf(v, L.ref_q, L.ref_e[i]);
}
template <typename T> __device__ __forceinline__ float to_store(const Lattice &L, int i, float d) {
    if constexpr (std::is_same<T, float>::value) return d;
    else return (d - L.ref_e[i]) * L.ref_iq;       // (one rounding: the scaling is exact)
}
struct Physics {
    float omega;                // 1 / tau
    float kf;                   // 1 - 1/(2 tau): prefactor of F_i (Eq. 15)
    float kforce;               // kf (Eq. 18 as printed) or 1 (momentum exchange)
    float phi_k2;               // -4 / (epsilon ln 2): phi = 1 / (1 + 2^(phi_k2 l)) = 1 / (1 + exp(-4 l / eps))
    float cut;                  // phi tail kept while l >= -cut
    int ck;                     // PS: half-width K of each particle's covered-area table (0: none)
    double cut_d;
};

// Tile bins.  A step reads the bins of its own positions and fills the next
// step's, so records come in two copies by step parity.  The counts rotate
// through three arrays: a step reads count[rot], its particle updates add to
// count[rot + 1], and it zeroes count[rot + 2], which nothing uses during the
// step, so that no pass of its own is needed to clear them.
struct Bins {                   // one step's view
    int *count;                 // per tile: particles binned (may exceed MAXC), or their mask (see slot_mask)
    int2 *ids;                  // per tile: MAXC (particle, index of the tile in the particle's list)
    float4 *rec;                // per tile and slot, 3 records: (cx_hi, cx_lo, cy_hi, cy_lo),
                                // (r, ux_hi, uy_hi, omega_hi), (ux_lo, uy_lo, omega_lo, packed
                                // floor(cx), floor(cy): 16 bits each)
    int *pslot;                 // per particle: MAXT tiles it reaches and its slots there (tile * MAXC + slot;
                                // -1: overflowed, or another strip's)
    int *npslot;                // per particle: tiles reached
    int *done;                  // per particle: minus the partials its update still waits for
};

// The step a lattice stands at, in device memory: fused steps advance it, so
// that launches recorded into a graph find it whatever ran before them.
// (Contexts without fused steps, a strip's and the static step's, have none:
// their counts rotate by parity.)
struct StepClock {
    unsigned tag;               // step number, marks the step's force partials
    int rot;                    // which of the three tile-count arrays the step reads
};

struct BinSet {
    int *count;                 // 3 arrays of `tiles`
    int2 *ids;                  // 2 x tiles x MAXC
    float4 *rec;                // 2 x tiles x MAXC x NREC
    int *pslot, *npslot, *done; // 2 x parts x MAXT, 2 x parts, 2 x parts
    float *cover;               // PS: per particle, the covered areas of the (2K+1)^2 cells about
                                // (floor X, floor Y), row-major; shared by both parities
    int tiles, parts;           // array strides
    int by_slot;                // the partials' layout, see partials_by_slot
};

// A particle's force partials, one per row of each tile it reaches, lie with
// the particle (MAXT tiles each, in the order of its list: 16 KB) or with the
// tile's slots (MAXC each: 4 KB a tile).  With the particle its update finds
// them without its list; with the slots many small discs take far less memory.
// (us per step in FP32 with the particle and by slot: 100 discs on 512^2 14.05
// and 14.5, 600 on 1024^2 30.5 and 31.4, 2000 on 2048^2 79.7 and 84.5, 20000 on
// 4096^2 455 and 460, 84000 there 1409 and 1421, where they take 1376 MB and 67
// MB.)  So by slot from one particle a tile on, where 16 KB each begin to count
// beside the tile's 74 KB of populations (37 KB in 16 bits).
__host__ __device__ inline bool partials_by_slot(long long tiles, long long parts) { return parts > 64 && parts > tiles; }
__host__ __device__ inline long long partial_entries(long long tiles, long long parts) {
    return (partials_by_slot(tiles, parts) ? tiles * MAXC : parts * MAXT) * TILE_H;
}

// The tile of a particle's list entry (Bins::pslot), or -1.
__device__ __forceinline__ int listed_tile(int w) { return w == -1 ? -1 : (int)((unsigned)w / MAXC); }

__host__ __device__ inline int rot3(int r) { return r >= 3 ? r - 3 : r; }

__host__ __device__ inline Bins bins_at(const BinSet &b, int par, int rot) {
    Bins v;
    const long long t = (long long)par * b.tiles, q = (long long)par * b.parts;
    v.count = b.count + (long long)rot * b.tiles;
    v.ids = b.ids + t * MAXC;
    v.rec = b.rec + t * MAXC * NREC;
    v.pslot = b.pslot + q * MAXT;
    v.npslot = b.npslot + q;
    v.done = b.done + q;
    return v;
}

// The slots a tile's count word `w` says are taken.  With at most MAXC
// particles a particle's slot is its number and the word is the mask itself,
// so binning sends an OR and waits for no answer; with more, slots are handed
// out by a counter, whose value may exceed MAXC.
__device__ __forceinline__ bool masked_bins(int np) { return np <= MAXC; }
__device__ __forceinline__ unsigned slot_mask(int w, int np) {
    if (masked_bins(np)) return (unsigned)w;
    return w >= MAXC ? 0xffffffffu : (1u << w) - 1u;
}

// ------------------------------------------------------------ small helpers
__device__ __forceinline__ int wrap_or_clamp(int v, int n, int periodic) {
    if (periodic) return v < 0 ? v + n : (v >= n ? v - n : v);
    return v < 0 ? 0 : (v >= n ? n - 1 : v);
}

// Row sy (in [-1, ny]) of plane i of the post-collision populations `src`:
// wrapped on a periodic axis, from a halo buffer across a strip's cut, else
// clamped (an edge row, whose pulled values the edge scheme replaces).
template <typename T>
__device__ __forceinline__ const T *plane_row(const T *src, const Lattice &L, int i, int sy) {
    if (sy < 0 && L.halo[0]) return static_cast<const T *>(L.halo[0]) + (long long)i * L.pitch;
    if (sy >= L.ny && L.halo[1]) return static_cast<const T *>(L.halo[1]) + (long long)i * L.pitch;
    return src + i * L.plane + (long long)wrap_or_clamp(sy, L.ny, L.per_y) * L.row;
}

// Populations of the form X_i = w_i [S + 3 c_i.B + 4.5 c_i^T M c_i] (the
// equilibrium of Eq. 2 has this form with B = rho u, M = rho u u^T; so has the
// collision's relaxation target plus force term of Eqs. 13 and 15), for a
// given zeroth moment m0 = sum_i X_i, so S = m0 - 1.5 tr M.
//
// The constants are chosen so that the moments come out exact for the FP32
// constants themselves: 4.5 w_1 = 1/2 and 4.5 w_5 = 1/8 are exact, the
// first-moment weights a1 ~ 1/3 and a5 = (1 - 2 a1) / 4 satisfy
// 2 a1 + 4 a5 = 1 exactly, and X_0 takes the remainder of m0.  Rounded
// weights would otherwise bias the momentum by ~1e-8 every step.
constexpr float W1F = 1.0f / 9.0f, W5F = 1.0f / 36.0f;
constexpr float A1F = 1.0f / 3.0f;
constexpr float A5F = (float)((1.0 - 2.0 * (double)A1F) / 4.0);

__device__ __forceinline__ void moment_form(float m0, float Bx, float By, float Mxx, float Myy, float Mxy, float X[9]) {
    const float S = fmaf(-1.5f, Mxx + Myy, m0);
    const float ax = fmaf(W1F, S, 0.5f * Mxx), ay = fmaf(W1F, S, 0.5f * Myy);
    const float tr = Mxx + Myy;
    const float ap = fmaf(W5F, S, 0.125f * fmaf(2.0f, Mxy, tr));
    const float am = fmaf(W5F, S, 0.125f * fmaf(-2.0f, Mxy, tr));
    const float bx = A1F * Bx, by = A1F * By, bp = A5F * (Bx + By), bm = A5F * (By - Bx);
    X[0] = fmaf(-2.0f, (ax + ay) + (ap + am), m0);
    X[1] = ax + bx; X[3] = ax - bx;
    X[2] = ay + by; X[4] = ay - by;
    X[5] = ap + bp; X[7] = ap - bp;
    X[6] = am + bm; X[8] = am - bm;
}

// Equilibrium deviation f^eq_i(rho, u) - w_i (Eq. 2), rho = 1 + drho.
__device__ __forceinline__ void eq_dev9(float drho, float rho, float ux, float uy, float X[9]) {
    const float rux = rho * ux, ruy = rho * uy;
    moment_form(drho, rux, ruy, rux * ux, ruy * uy, rux * uy, X);
}

// Collision of Eq. 13 with f^eq of Eq. 2 (corrected velocity, Eq. 17) and the
// force term of Eq. 15, in deviation form:
//   d'_i = d_i + (X_i - omega d_i),  X_i = omega d^eq_i + phi F_i,
// and X has the form w_i [S + 3 c_i.B + 4.5 c_i^T M c_i] with
//   B = omega rho u + k (u_s - u*),  M = omega rho u u^T + k (u_s u_s^T - u* u*^T),
//   sum_i X_i = omega (rho - 1),     k = (1 - 1/2tau) rho phi,
// which is Eqs. 2 and 15 summed and regrouped by powers of c_i.  Because
// rho u = j + phi rho (u_s - u*) / 2 (Eq. 17) and omega/2 + (1 - 1/2tau) = 1,
// B = omega j + phi rho (u_s - u*): the momentum handed to the fluid is formed
// without dividing by rho, so no rounding of j / rho biases it.  The force
// part of M is formed from (u_s - u*) and (u_s + u*) rather than as a
// difference of squares.  Nodes go in pairs on the paired FP32 instructions
// of sm_100+ (each component rounds exactly as the scalar op).
__device__ __forceinline__ float2 f2(float a) { return make_float2(a, a); }
__device__ __forceinline__ float2 add2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 mul2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 fma2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
// a - b in one paired instruction: b * -1 + a rounds once, as a - b does.  (The
// paired add has no subtracting form: negating b first takes two more.)
__device__ __forceinline__ float2 sub2(float2 a, float2 b) { return fma2(b, f2(-1.0f), a); }
__device__ __forceinline__ float2 neg2(float2 a) { return mul2(a, f2(-1.0f)); }

__device__ __forceinline__ void moment_form2(float2 m0, float2 Bx, float2 By, float2 Mxx, float2 Myy, float2 Mxy,
                                             float2 X[9]) {
    const float2 tr = add2(Mxx, Myy);
    const float2 S = fma2(f2(-1.5f), tr, m0);
    const float2 ax = fma2(f2(W1F), S, mul2(f2(0.5f), Mxx)), ay = fma2(f2(W1F), S, mul2(f2(0.5f), Myy));
    const float2 ap = fma2(f2(W5F), S, mul2(f2(0.125f), fma2(f2(2.0f), Mxy, tr)));
    const float2 am = fma2(f2(W5F), S, mul2(f2(0.125f), fma2(f2(-2.0f), Mxy, tr)));
    const float2 bx = mul2(f2(A1F), Bx), by = mul2(f2(A1F), By);
    const float2 bp = mul2(f2(A5F), add2(Bx, By)), bm = mul2(f2(A5F), sub2(By, Bx));
    X[0] = fma2(f2(-2.0f), add2(add2(ax, ay), add2(ap, am)), m0);
    X[1] = add2(ax, bx); X[3] = sub2(ax, bx);
    X[2] = add2(ay, by); X[4] = sub2(ay, by);
    X[5] = add2(ap, bp); X[7] = sub2(ap, bp);
    X[6] = add2(am, bm); X[8] = sub2(am, bm);
}

// d + (X - omega d): the small change is rounded on its own before it is
// added (a single fma((1 - omega), d, X) measured ~15% larger errors against
// the FP64 oracle on wall-driven flow).
__device__ __forceinline__ void relax2(float2 d[9], float omega, const float2 X[9]) {
#pragma unroll
    for (int i = 0; i < 9; ++i) d[i] = add2(d[i], fma2(f2(-omega), d[i], X[i]));
}

// The collision acts on the stored values.  FP32 stores d_i itself.  16-bit
// storage holds s_i = (d_i - e_i) / q, and since e_i has the moment form
// with the reference moments (m0e, Be, Me) and q is a power of two,
//   s'_i = s_i + (Y_i - omega s_i),  Y = (X - omega e) / q,
// where Y is the moment form of (omega sum s, (B - omega Be) / q,
// (M - omega Me) / q): the zeroth input is omega times the stored values'
// own sum, the first moment's part omega j becomes omega times the stored
// first moment, and only M, a product of the physical moments, needs the
// reference subtracted.  (ms, jxs, jys are the moments of the stored values.)
template <typename T>
__device__ __forceinline__ void relax_to2(float2 d[9], const Lattice &L, float omega, float2 ms, float2 Bxs,
                                          float2 Bys, float2 Mxx, float2 Myy, float2 Mxy) {
    const float2 om = f2(omega);
    if constexpr (!std::is_same<T, float>::value) {
        const float2 iq = f2(L.ref_iq);
        Mxx = mul2(add2(Mxx, f2(-(omega * L.ref_m[3]))), iq);
        Myy = mul2(add2(Myy, f2(-(omega * L.ref_m[4]))), iq);
        Mxy = mul2(add2(Mxy, f2(-(omega * L.ref_m[5]))), iq);
    }
    float2 X[9];
    moment_form2(mul2(om, ms), Bxs, Bys, Mxx, Myy, Mxy, X);
    relax2(d, omega, X);
}

// phi = 0 (plain BGK of Eq. 1): B = omega j and, as rho u = j,
// M = omega rho u u^T = B u^T.
template <typename T>
__device__ __forceinline__ void collide_plain2(float2 d[9], const Lattice &L, float omega, float2 ms, float2 jxs,
                                               float2 jys, float2 jx, float2 jy, float2 ux, float2 uy) {
    const float2 om = f2(omega);
    const float2 Bx = mul2(om, jx), By = mul2(om, jy);
    if constexpr (std::is_same<T, float>::value)
        relax_to2<T>(d, L, omega, ms, Bx, By, mul2(Bx, ux), mul2(By, uy), mul2(Bx, uy));
    else
        relax_to2<T>(d, L, omega, ms, mul2(om, jxs), mul2(om, jys), mul2(Bx, ux), mul2(By, uy), mul2(Bx, uy));
}

template <typename T>
__device__ __forceinline__ void collide2(float2 d[9], const Lattice &L, float omega, float2 ms, float2 jxs,
                                         float2 jys, float2 rho, float2 ux, float2 uy, float2 kphi, float2 prho,
                                         float2 dux, float2 duy, float2 usx, float2 usy, float2 uax, float2 uay) {
    const float2 om = f2(omega);
    const float2 orho = mul2(om, rho);
    float2 px = mul2(prho, dux), py = mul2(prho, duy);
    if constexpr (!std::is_same<T, float>::value) {
        px = mul2(px, f2(L.ref_iq));
        py = mul2(py, f2(L.ref_iq));
    }
    const float2 Bxs = fma2(om, jxs, px), Bys = fma2(om, jys, py);
    const float2 rux = mul2(orho, ux);
    const float2 Mxx = fma2(rux, ux, mul2(kphi, mul2(dux, add2(usx, uax))));
    const float2 Myy = fma2(mul2(orho, uy), uy, mul2(kphi, mul2(duy, add2(usy, uay))));
    const float2 Mxy = fma2(rux, uy, mul2(kphi, fma2(dux, usy, mul2(uax, duy))));
    relax_to2<T>(d, L, omega, ms, Bxs, Bys, Mxx, Myy, Mxy);
}

// Tile ranges along one axis covered by [X - R, X + R] (a disc's bounding
// interval); periodic intervals wrap and may split in two.  Shared by the
// binning and the reduction so both visit the same tiles in the same order.
struct AxisTiles {
    int n;
    int lo[2], hi[2];
};

// floor and ceil to int (one instruction on the device), and v mod n for v
// mostly within one period of [0, n).
__host__ __device__ inline int floor_int(double v) {
#ifdef __CUDA_ARCH__
    return __double2int_rd(v);
#else
    return (int)floor(v);
#endif
}
__host__ __device__ inline int ceil_int(double v) {
#ifdef __CUDA_ARCH__
    return __double2int_ru(v);
#else
    return (int)ceil(v);
#endif
}
__host__ __device__ inline int wrap_int(int v, int n) {
    if (v >= -n && v < 0) return v + n;
    if (v >= n && v - n < n) return v - n;
    if (v >= 0 && v < n) return v;
    return ((v % n) + n) % n;
}

// (tiles of 2^shift nodes)
__host__ __device__ inline AxisTiles axis_tiles(double X, double R, int n, int shift, int ntiles, int periodic) {
    AxisTiles t;
    int il = floor_int(X - R), ih = ceil_int(X + R);
    if (periodic) {
        if (ih - il + 1 >= n) { t.n = 1; t.lo[0] = 0; t.hi[0] = ntiles - 1; return t; }
        const int a = wrap_int(il, n), b = wrap_int(ih, n);
        if (a <= b) { t.n = 1; t.lo[0] = a >> shift; t.hi[0] = b >> shift; return t; }
        int first_hi = b >> shift, second_lo = a >> shift;
        if (first_hi >= second_lo) { t.n = 1; t.lo[0] = 0; t.hi[0] = ntiles - 1; return t; }
        t.n = 2; t.lo[0] = 0; t.hi[0] = first_hi; t.lo[1] = second_lo; t.hi[1] = ntiles - 1;
        return t;
    }
    il = il < 0 ? 0 : il;
    ih = ih > n - 1 ? n - 1 : ih;
    if (il > ih) { t.n = 0; return t; }
    t.n = 1; t.lo[0] = il >> shift; t.hi[0] = ih >> shift;
    return t;
}

// ------------------------------------------------------------ async copies
__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_fence_init() {
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes) : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t parity) {
    uint32_t ok;
    asm volatile(
        "{\n\t.reg .pred p;\n\t"
        "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    return ok != 0;
}

__device__ __forceinline__ unsigned long long global_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Wait for a phase of an mbarrier, giving up after WAIT_LIMIT_NS.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, uint32_t parity) {
    if (mbar_try_wait(bar, parity)) return true;
    const unsigned long long t0 = global_ns();
    for (;;) {
        if (mbar_try_wait(bar, parity)) return true;
        if (global_ns() - t0 > WAIT_LIMIT_NS) return false;
    }
}

// Order this thread's earlier shared-memory reads before later writes of the
// async proxy (the bulk copies) to the same buffer.
__device__ __forceinline__ void fence_proxy_async_smem() {
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}

__device__ __forceinline__ void bulk_copy_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_u32(dst)), "l"(src), "r"(bytes), "r"(smem_u32(bar))
                 : "memory");
}

// Stage the nine source rows of row segment (row y, segment tx):
// plane i comes from row y - c_iy, columns [tx*128 - halo, tx*128 + 128 + halo).
// Lane 0 arms the barrier with the byte count, lanes 0..8 issue one copy each.
// The population buffers carry GUARD readable elements before and after, so
// the copies of edge segments stay inside the allocation.
template <typename T>
__device__ __forceinline__ void issue_segment(const T *__restrict__ src, const Lattice &L, int y, int tx, T *stage,
                                              uint64_t *bar, int lane) {
    constexpr int H = halo_of<T>(), SW = segw_of<T>();
    if (lane == 0) mbar_expect_tx(bar, 9u * SW * sizeof(T));
    __syncwarp();
    if (lane < 9) {
        const T *g = plane_row<T>(src, L, lane, y - cyof(lane)) + (tx * TILE_W - H);
        bulk_copy_g2s(stage + lane * SW, g, SW * sizeof(T), bar);
    }
}

// Periodic x: the staged halo of a row's first segment does not hold column
// nx - 1 (what node 0 streams from in the three directions with c_ix = +1),
// nor does the stage of its last segment hold column 0 after column nx - 1
// (what node nx - 1 streams from with c_ix = -1).  When a warp issues such a
// segment's copy, lanes 0..2 also load the first value (planes 1, 5, 8) and
// lanes 3..5 the second (planes 3, 6, 7), raw; once the copy has landed,
// wrap_patch writes them where the pulls look.  wrap_lane_plane gives the
// plane of the lane's value and whether the segment needs it.
__device__ __forceinline__ int wrap_lane_plane(const Lattice &L, int tx, int lane) {
    if (!L.per_x || lane >= 6) return -1;
    const bool first = tx == 0, last = tx * TILE_W + TILE_W >= L.nx;
    if (lane < 3) return first ? (lane == 0 ? 1 : (lane == 1 ? 5 : 8)) : -1;
    return last ? (lane == 3 ? 3 : (lane == 4 ? 6 : 7)) : -1;
}

template <typename T>
__device__ __forceinline__ T wrap_load(const T *__restrict__ src, const Lattice &L, int y, int tx, int lane) {
    const int i = wrap_lane_plane(L, tx, lane);
    if (i < 0) return T();
    const T *row = plane_row<T>(src, L, i, y - cyof(i));
    return __ldcg(row + (lane < 3 ? L.nx - 1 : 0));
}

template <typename T>
__device__ __forceinline__ void wrap_patch(T *stage, const Lattice &L, int tx, int lane, T v) {
    constexpr int H = halo_of<T>(), SW = segw_of<T>();
    const int i = wrap_lane_plane(L, tx, lane);
    if (i >= 0) stage[i * SW + (lane < 3 ? H - 1 : H + (L.nx - tx * TILE_W))] = v;
}

// Non-equilibrium extrapolation at an edge node (x, y) (Guo et al. 2002, as
// the paper's Sec. 3 uses): d_b = deq(rho_b, u_b) + d_n - deq(rho_n, u_n),
// with n the inner neighbour (diagonal at corners; corners take the
// south/north condition).
// d_b from the inner neighbour's streamed values dn and the side's condition.
__device__ __forceinline__ void extrapolate(const Lattice &L, int side, const float dn[9], float out[9]) {
    float drn = 0.f, jx = 0.f, jy = 0.f;
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        drn += dn[i];
        jx += cxof(i) * dn[i];
        jy += cyof(i) * dn[i];
    }
    const float rhon = 1.0f + drn;
    const float unx = jx / rhon, uny = jy / rhon;
    // select the side's parameters without indexing the kernel-parameter arrays
    int kind = L.side_kind[0];
    float sux = L.side_ux[0], suy = L.side_uy[0], sdr = L.side_drho[0];
#pragma unroll
    for (int k = 1; k < 4; ++k)
        if (side == k) { kind = L.side_kind[k]; sux = L.side_ux[k]; suy = L.side_uy[k]; sdr = L.side_drho[k]; }
    float drb, ubx, uby;
    if (kind == SIDE_VELOCITY) {
        drb = drn; ubx = sux; uby = suy;
    } else {
        drb = sdr; ubx = unx; uby = uny;
    }
    // f^eq(rho_b, u_b) - f^eq(rho_n, u_n) is linear in the moments, so it is
    // the moment form of the moment differences, formed without cancellation:
    // with d = rho_b - rho_n and v = u_b - u_n,
    //   rho_b u_b - rho_n u_n = d u_b + rho_n v,
    //   rho_b u_b u_b - rho_n u_n u_n = d u_b u_b + rho_n (v (u_b + u_n))   (xx, yy),
    //   rho_b ubx uby - rho_n unx uny = d ubx uby + rho_n (vx uby + unx vy).
    const float d = drb - drn, vx = ubx - unx, vy = uby - uny;
    const float Bx = fmaf(d, ubx, rhon * vx), By = fmaf(d, uby, rhon * vy);
    const float Mxx = fmaf(d * ubx, ubx, rhon * (vx * (ubx + unx)));
    const float Myy = fmaf(d * uby, uby, rhon * (vy * (uby + uny)));
    const float Mxy = fmaf(d * ubx, uby, rhon * fmaf(vx, uby, unx * vy));
    float X[9];
    moment_form(d, Bx, By, Mxx, Myy, Mxy, X);
#pragma unroll
    for (int i = 0; i < 9; ++i) out[i] = dn[i] + X[i];
}

// The row whose streamed values row y's sweep starts from: an edge row's nodes
// extrapolate from their inner neighbours (the same column one row in; corners
// diagonally), so an edge row stages its neighbour's source rows.
template <bool EDGES>
__device__ __forceinline__ int streamed_row(const Lattice &L, int y) {
    if (EDGES && south_edge_row(L, y)) return 1;
    if (EDGES && north_edge_row(L, y)) return L.ny - 2;
    return y;
}

// ------------------------------------------------------------ PS-LBM solid fraction
// The paper's comparison method (PS-LBM, Sec. 2.2) weights its collision by
// B = eps_s (Eq. 8), the area of the node's unit cell covered by the solid.
// cell_cover returns the area of [dx - 1/2, dx + 1/2] x [dy - 1/2, dy + 1/2]
// inside the disc of radius r >= 1 centred at the origin: the shoelace area
// of the polygon formed, counter-clockwise, by the corners inside the disc
// and the points where the circle crosses the cell edges, plus the circular
// segment between each chord that polygon draws across the circle and its
// arc.  The polygon is summed in the cell's own frame (coordinates of size
// 1/2, so FP32 keeps ~1e-6).  Each corner is classified once (inside:
// distance < r) and every edge takes its crossings from the classes of its
// two ends (one crossing where they differ; none or two where both are
// outside), so a corner on the circle, seen by two edges, cannot be counted
// twice or lost.  For r >= 1 every arc inside a unit cell is a minor arc.
// Both routines stay out of line: inlined into the sweep's four node slots
// they evict the sweep's own code from the instruction cache.
static __device__ __noinline__ float segment_area(float ex, float ey, float ix, float iy, float r, float rinv) {
    // area between the chord E-I and the minor arc: r^2 (asin s - s sqrt(1 - s^2)), s = |EI| / 2r
    const float s = 0.5f * sqrtf((ix - ex) * (ix - ex) + (iy - ey) * (iy - ey)) * rinv;
    float g;
    if (s < 0.3f) {     // Taylor series: 2/3 s^3 + 1/5 s^5 + 3/28 s^7 + 5/72 s^9 + 35/704 s^11
        const float s2 = s * s;
        g = s * s2 * (2.0f / 3.0f + s2 * (0.2f + s2 * (3.0f / 28.0f + s2 * (5.0f / 72.0f + s2 * (35.0f / 704.0f)))));
    } else {
        g = asinf(s) - s * sqrtf((1.0f - s) * (1.0f + s));
    }
    return r * r * g;
}

// The polygon and segment sums of cell_cover, fed one boundary point at a
// time in counter-clockwise order.
struct CoverWalk {
    float r, rinv;
    float area2 = 0.f, seg = 0.f;
    float fx = 0.f, fy = 0.f, lx = 0.f, ly = 0.f;   // first and last polygon vertex
    float ex = 0.f, ey = 0.f, ix0 = 0.f, iy0 = 0.f; // pending exit; first entry seen before any exit
    bool any = false, pending = false, first_entry = false;

    __device__ __forceinline__ void vertex(float vx, float vy) {
        if (any) area2 += lx * vy - vx * ly;
        else { fx = vx; fy = vy; any = true; }
        lx = vx; ly = vy;
    }
    __device__ __forceinline__ void entry(float vx, float vy) {
        if (pending) { seg += segment_area(ex, ey, vx, vy, r, rinv); pending = false; }
        else if (!first_entry) { first_entry = true; ix0 = vx; iy0 = vy; }
        vertex(vx, vy);
    }
    __device__ __forceinline__ void exit(float vx, float vy) {
        vertex(vx, vy);
        ex = vx; ey = vy; pending = true;
    }
};

// Half the chord the circle cuts on a line at distance |p| from the centre.
__device__ __forceinline__ float half_chord(float p, float r) {
    const float a = fabsf(p);
    return sqrtf(fmaxf((r - a) * (r + a), 0.f));
}

__device__ __forceinline__ float clampf(float v, float lo, float hi) { return fminf(fmaxf(v, lo), hi); }

static __device__ __noinline__ float cell_cover(float dx, float dy, float r) {
    // the cell's extent about the disc centre; corners 0..3 counter-clockwise
    // from (x0, y0), edge k from corner k to corner k + 1
    const float x0 = dx - 0.5f, x1 = dx + 0.5f, y0 = dy - 0.5f, y1 = dy + 0.5f;
    const float r2 = r * r;
    const float xx0 = x0 * x0, xx1 = x1 * x1, yy0 = y0 * y0, yy1 = y1 * y1;
    const bool in0 = xx0 + yy0 < r2, in1 = xx1 + yy0 < r2, in2 = xx1 + yy1 < r2, in3 = xx0 + yy1 < r2;
    // both ends outside: the circle crosses twice iff the foot of the
    // perpendicular from the centre lies inside the edge and |p| < r
    const bool mx = x0 < 0.f && 0.f < x1, my = y0 < 0.f && 0.f < y1;
    CoverWalk w;
    w.r = r;
    w.rinv = __frcp_rn(r);

    // edge 0: y = y0, x rising; enters at x = -h, leaves at x = +h
    if (in0) w.vertex(-0.5f, -0.5f);
    {
        const bool two = !in0 && !in1 && mx && fabsf(y0) < r;
        const bool en = !in0 && (in1 || two), ex = !in1 && (in0 || two);
        if (en || ex) {
            const float h = half_chord(y0, r);
            if (en) w.entry(clampf(-h, x0, x1) - dx, -0.5f);
            if (ex) w.exit(clampf(h, x0, x1) - dx, -0.5f);
        }
    }
    // edge 1: x = x1, y rising; enters at y = -h, leaves at y = +h
    if (in1) w.vertex(0.5f, -0.5f);
    {
        const bool two = !in1 && !in2 && my && fabsf(x1) < r;
        const bool en = !in1 && (in2 || two), ex = !in2 && (in1 || two);
        if (en || ex) {
            const float h = half_chord(x1, r);
            if (en) w.entry(0.5f, clampf(-h, y0, y1) - dy);
            if (ex) w.exit(0.5f, clampf(h, y0, y1) - dy);
        }
    }
    // edge 2: y = y1, x falling; enters at x = +h, leaves at x = -h
    if (in2) w.vertex(0.5f, 0.5f);
    {
        const bool two = !in2 && !in3 && mx && fabsf(y1) < r;
        const bool en = !in2 && (in3 || two), ex = !in3 && (in2 || two);
        if (en || ex) {
            const float h = half_chord(y1, r);
            if (en) w.entry(clampf(h, x0, x1) - dx, 0.5f);
            if (ex) w.exit(clampf(-h, x0, x1) - dx, 0.5f);
        }
    }
    // edge 3: x = x0, y falling; enters at y = +h, leaves at y = -h
    if (in3) w.vertex(-0.5f, 0.5f);
    {
        const bool two = !in3 && !in0 && my && fabsf(x0) < r;
        const bool en = !in3 && (in0 || two), ex = !in0 && (in3 || two);
        if (en || ex) {
            const float h = half_chord(x0, r);
            if (en) w.entry(-0.5f, clampf(h, y0, y1) - dy);
            if (ex) w.exit(-0.5f, clampf(-h, y0, y1) - dy);
        }
    }
    if (!w.any) return 0.f;
    w.area2 += w.lx * w.fy - w.fx * w.ly;
    if (w.pending && w.first_entry) w.seg += segment_area(w.ex, w.ey, w.ix0, w.iy0, r, w.rinv);
    return 0.5f * w.area2 + w.seg;
}

// 16 bytes from global to shared memory without a register in between.
__device__ __forceinline__ void copy16_async(void *dst, const void *src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(smem_u32(dst)), "l"(src) : "memory");
}
__device__ __forceinline__ void copies_async_done() { asm volatile("cp.async.wait_all;" ::: "memory"); }

// ------------------------------------------------------------ the sweep
// Mode: STEP writes the collided populations and the force partials; FIELDS
// writes rho, the corrected velocity and phi of the streamed state instead.
enum : int { MODE_STEP = 0, MODE_FIELDS = 1 };

struct FieldsOut {
    float *rho, *ux, *uy, *phi;   // dense [ny][nx]
};

struct PartArgs;

// Everything one lattice's sweep needs.
template <typename T>
struct SweepArgs {
    T *buf[2];                  // populations by step parity (GUARD elements in)
    Lattice L;
    Physics ph;
    BinSet B;                   // tile bins (np > 0)
    float4 *partial;            // force / torque partials and tag: per particle, tile of its list and row (or by slot)
    int *err;                   // the lattice's error word
    const PartArgs *pa;         // the particle update's arguments (device memory; batches)
    StepClock *clock;           // (null: see StepClock)
    int np;                     // particles (0: no bins to read)
    // A segment's candidate records are loaded beside the word that says which
    // are there (not after it: a trip to the L2 less) where particles own their
    // slots and discs times segments are at most 4096: records that no node uses
    // are loaded too.  (us per step without and with it, FP32, by discs x
    // segments: 200, 8.42 and 8.34; 2048 to 8000, within 0.1 either way; 24576,
    // 11.0 and 11.2; 65536, 11.4 and 11.7; 1048576, 49.7 and 59.5.)
    bool eager;
    // Every second step takes the segments from the end, where two buffers do
    // not fit the L2: the rows a step wrote last are read first by the next one
    // and are still there.  (4096^2, us per step: FP32 216 -> 214, PS 238 ->
    // 235; the 400 x 2000 box, which fits, lost 0.2 of 16.)
    bool turn;
    int cur;                    // parity of the launch's first step
    unsigned ntx_inv;           // floor(2^32 / ntx) + 1 (saturated), see row_of
};

// A batched sweep walks one work list over many lattices, their descriptors
// held in the kernel's parameter space (uniform constant-cache reads, no
// aliasing with the stores): lattice k owns row segments
// [item_start[k], item_start[k+1]) and tiles [tile_start[k], tile_start[k+1]).
constexpr int BATCH_LAUNCH_MAX = 84;     // lattices per batched launch

template <typename T>
struct BatchArgs {
    SweepArgs<T> a[BATCH_LAUNCH_MAX];
    int item_start[BATCH_LAUNCH_MAX + 1];
    int tile_start[BATCH_LAUNCH_MAX + 1];
    int part_start[BATCH_LAUNCH_MAX + 1];
    int n;
};
static_assert(sizeof(BatchArgs<float>) <= 32000, "batched sweep parameters exceed the parameter space");

// Largest k with start[k] <= v (start[0] = 0, start ascending, n entries + 1).
template <typename P>
__device__ __forceinline__ int batch_find(const P &start, int n, int v) {
    int lo = 0, hi = n - 1;
    while (lo < hi) {
        const int mid = (lo + hi + 1) >> 1;
        if (start[mid] <= v) lo = mid; else hi = mid - 1;
    }
    return lo;
}

// Per-warp state of the staged segment.
struct Ring {
    uint64_t *bar;
    uint32_t parity;            // phase parity the next wait expects
    bool pending;               // copies in flight
};

// A contribution to a particle is counted without ordering the count after the
// contribution: a release would wait for every store the warp has in flight (a
// segment's 9 x 128 populations).  Each partial instead carries its step's tag
// in the same 16-byte store, and whoever finds the count complete reads the
// partials until their tags are there.
__device__ __forceinline__ void count_done(int *counter) {
    asm volatile("red.add.relaxed.gpu.global.s32 [%0], 1;" ::"l"(counter) : "memory");
}
__device__ __forceinline__ int load_done(const int *counter) {
    int v;
    asm volatile("ld.relaxed.gpu.global.s32 %0, [%1];" : "=r"(v) : "l"(counter) : "memory");
    return v;
}
__device__ __forceinline__ void store_partial(float4 *p, float x, float y, float z, unsigned tag) {
    asm volatile("{\n\t.reg .b64 a, b;\n\t.reg .b128 v;\n\t"
                 "mov.b64 a, {%1, %2};\n\tmov.b64 b, {%3, %4};\n\tmov.b128 v, {a, b};\n\t"
                 "st.relaxed.gpu.global.b128 [%0], v;\n\t}"
                 ::"l"(p), "r"(__float_as_uint(x)), "r"(__float_as_uint(y)), "r"(__float_as_uint(z)), "r"(tag)
                 : "memory");
}
__device__ __forceinline__ float4 load_partial(const float4 *p) {
    uint32_t x, y, z, w;
    asm volatile("{\n\t.reg .b64 a, b;\n\t.reg .b128 v;\n\t"
                 "ld.relaxed.gpu.global.b128 v, [%4];\n\tmov.b128 {a, b}, v;\n\t"
                 "mov.b64 {%0, %1}, a;\n\tmov.b64 {%2, %3}, b;\n\t}"
                 : "=r"(x), "=r"(y), "=r"(z), "=r"(w)
                 : "l"(p)
                 : "memory");
    return make_float4(__uint_as_float(x), __uint_as_float(y), __uint_as_float(z), __uint_as_float(w));
}

// The streamed value f_i(x) = f'_i(x - c_i) of plane i at node e of the
// staged segment (e in [-1, TILE_W]: the 16-byte halos hold the neighbours).
template <typename T, int I>
__device__ __forceinline__ float staged_pull(const Lattice &L, const T *stage, int e) {
    constexpr int H = halo_of<T>(), SW = segw_of<T>();
    return from_store<T>(L, I, Storage<T>::lds1(stage + I * SW + H + e - cxof(I)));
}

template <typename T, int I = 0>
__device__ __forceinline__ void staged_pull9(const Lattice &L, const T *stage, int e, float out[9]) {
    out[I] = staged_pull<T, I>(L, stage, e);
    if constexpr (I < 8) staged_pull9<T, I + 1>(L, stage, e, out);
}

// The hardware's base-2 exponential and reciprocal (PTX ex2.approx, rcp.approx;
// subnormal results flush to zero, so 2^x for very negative x is 0).
__device__ __forceinline__ float ex2_approx(float x) {
    float r;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rcp_approx(float x) {
    float r;
    asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}
__device__ __forceinline__ float rsqrt_approx(float x) {
    float r;
    asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
    return r;
}

// 1 / v of a pair of densities: the hardware's approximation and one
// Newton-Raphson correction with its residual formed exactly by an FMA, after
// which the reciprocal is correctly rounded (Markstein, IBM J. Res. Dev. 34
// (1990) 111).  Compared with __frcp_rn over every normal FP32 value whose
// reciprocal is normal: the same bits.
__device__ __forceinline__ float2 recip2(float2 v) {
    const float2 r = make_float2(rcp_approx(v.x), rcp_approx(v.y));
    const float2 e = fma2(neg2(v), r, f2(1.0f));
    return fma2(r, e, r);
}

// Square roots of a pair of squared distances (0, or at least the square of
// a distance's rounding), the same way: v rsqrt(v), then one Newton-Raphson
// (Heron) correction by the exact residual.
__device__ __forceinline__ float2 sqrt2(float2 v) {
    const float2 q = make_float2(rsqrt_approx(fmaxf(v.x, 1e-30f)), rsqrt_approx(fmaxf(v.y, 1e-30f)));
    const float2 s = mul2(v, q);
    const float2 e = fma2(neg2(s), s, v);
    return fma2(e, mul2(f2(0.5f), q), s);
}

// Slot m (0 or 1) of a node pair.
__device__ __forceinline__ float &slot(float2 &v, int m) { return m ? v.y : v.x; }

// Two neighbouring warps that share a segment (run_steps, HALVES) meet.
__device__ __forceinline__ void meet_partner() {
    asm volatile("bar.sync %0, 64;" ::"r"(1 + (int)(threadIdx.x >> 6)) : "memory");
}

// One row segment (row y, segment tx) of lattice A, populations src -> dst,
// bins B: wait for its staged rows (and write in the periodic-edge values wv,
// see wrap_load), then sweep its 128 nodes in two passes of 64 (lane l takes
// nodes 2l and 2l + 1 of each half, so every store of a pass is one
// contiguous run per plane), hand the stage to the next segment (row ny2,
// segment nx2 of lattice Ln, populations srcn; its edge values go to wv) once
// the second pass has read it, and sum the segment's force / torque per
// candidate particle.  FUSED: also count the contributions, marked with the
// step's tag (`count` false: not counted); HALVES: this warp runs the pass
// `half`, its neighbour the other.  Returns false if the bounded wait gave up.
template <typename T, int MODE, bool EDGES, bool PS, bool FUSED, bool HALVES = false>
__device__ __forceinline__ bool sweep_segment(const SweepArgs<T> &A, const T *src, T *dst, const Bins &B, int y, int tx,
                                              T *stage, Ring &ring, bool has_next, const T *srcn, const Lattice &Ln,
                                              int ny2, int nx2, float4 *crec, int *cid, T &wv, unsigned tag,
                                              bool count, const FieldsOut &fo, int lane, int half = 0) {
    constexpr int H = halo_of<T>(), SW = segw_of<T>();
    const Lattice &L = A.L;
    const Physics &ph = A.ph;
    const int ty = y / TILE_H, tile = ty * L.ntx + tx;
    const int tx0 = tx * TILE_W, ty0 = ty * TILE_H;

    // ---- the tile's candidate particles (records written by the binning),
    // loaded before the wait so that their latency overlaps it
    __syncwarp();
    unsigned cands = 0u;                    // the slots taken
    if (A.np > 0) {
        const long long r = (long long)tile * MAXC + lane;
        int2 mine = make_int2(-1, 0);       // the slot's particle, index of this tile in that particle's list
        auto fetch = [&]() {
#pragma unroll
            for (int q = 0; q < NREC; ++q) copy16_async(crec + q * MAXC + lane, B.rec + NREC * r + q);
            mine = __ldcg(B.ids + r);
        };
        const bool eager = A.eager && lane < A.np;
        if (eager) fetch();                 // (a slot not taken: stale, not used)
        cands = slot_mask(__ldcg(B.count + tile), A.np);
        if (!eager && (cands >> lane & 1u)) fetch();
        // beside the records: the particle, and the segment's force / torque on
        // it so far (first pass, then second pass added) with the index
        cid[lane] = mine.x;
        crec[NREC * MAXC + lane] = make_float4(0.f, 0.f, 0.f, __int_as_float(mine.y));
        copies_async_done();
    }

    // ---- wait for the staged rows
    // a warp-uniform decision: every lane leaves together if any gave up
    if (!__all_sync(0xffffffffu, mbar_wait_bounded(ring.bar, ring.parity))) {
        if (HALVES) meet_partner();
        return false;
    }
    ring.parity ^= 1u;
    ring.pending = false;

    const bool row_edge = EDGES && (south_edge_row(L, y) || north_edge_row(L, y));
    const bool col_edge = EDGES && !L.per_x && (tx == 0 || tx0 + TILE_W >= L.nx);
    if (L.per_x && (tx == 0 || tx0 + TILE_W >= L.nx)) wrap_patch<T>(stage, L, tx, lane, wv);
    // west / east edge nodes of a row that is not itself an edge row: the
    // non-equilibrium extrapolation from the inner neighbour's streamed values
    // (same row, staged).  Pull streaming reads each staged value at exactly
    // one node, so in FP32 storage lane 0 (west) and lane 1 (east) write the
    // edge node's extrapolated populations into the cells that node's pulls
    // read, and the pulls below pick them up.  (For nx >= 3 the cells one
    // edge writes and those the other reads are distinct.)  16-bit storage
    // would round them on the way; there the passes replace the pulled values.
    constexpr bool EDGE_IN_STAGE = std::is_same<T, float>::value;
    if (EDGE_IN_STAGE && col_edge && !row_edge && lane < 2) {
        const int xm = lane == 0 ? 0 : L.nx - 1;
        const int e = xm - tx0;
        if (e >= 0 && e < TILE_W) {
            float dn[9], ev[9];
            staged_pull9<T>(L, stage, e + (lane == 0 ? 1 : -1), dn);
            extrapolate(L, lane == 0 ? WEST : EAST, dn, ev);
#pragma unroll
            for (int i = 0; i < 9; ++i) Storage<T>::store1(stage + i * SW + H + e - cxof(i), to_store<T>(L, i, ev[i]));
        }
    }
    __syncwarp();   // candidate records and edge values visible to the whole warp

    unsigned badmax = 0u;

    // a row's last segment may end within its first half: its second pass
    // would hold no node (no store, no force share), so it is not run
    const int npass = tx0 + TILE_W / 2 < L.nx && !(HALVES && half == 0) ? 2 : 1;
#pragma unroll 1
    for (int pass = HALVES ? half : 0; pass < npass; ++pass) {
        const int e = pass * (TILE_W / 2) + 2 * lane;    // the pair's first node within the segment
        const int x = tx0 + e;

        // ---- pull-stream from the staged rows: f_i(x, t+1) = f'_i(x - c_i, t)
        float2 dk[9];
#pragma unroll
        for (int i = 0; i < 9; ++i) {
            const T *row = stage + i * SW + H + e;
            if (cxof(i) == 0) dk[i] = Storage<T>::lds2(row);
            else dk[i] = make_float2(Storage<T>::lds1(row - cxof(i)), Storage<T>::lds1(row + 1 - cxof(i)));
        }
        if constexpr (!EDGE_IN_STAGE) {
            if (col_edge && !row_edge) {
#pragma unroll
                for (int m = 0; m < 2; ++m) {
                    const int xm = x + m;
                    if (xm != 0 && xm != L.nx - 1) continue;
                    float dn[9], ev[9];
                    staged_pull9<T>(L, stage, e + m + (xm == 0 ? 1 : -1), dn);
                    extrapolate(L, xm == 0 ? WEST : EAST, dn, ev);
#pragma unroll
                    for (int i = 0; i < 9; ++i) slot(dk[i], m) = to_store<T>(L, i, ev[i]);
                }
            }
        }
        if (EDGES && row_edge) {
            // south / north edge rows (corners included): the stage holds the
            // neighbour row's pulls.  (Read from global memory, node by node
            // out of line, such a row took a warp 10 us, and the 400 x 2000
            // box's step waited 20 us for its two.)
#pragma unroll 1
            for (int m = 0; m < 2; ++m) {
                const int xm = x + m;
                if (xm >= L.nx) continue;
                const int in = L.per_x ? 0 : (xm == 0 ? 1 : (xm == L.nx - 1 ? -1 : 0));
                float dn[9], ev[9];
                staged_pull9<T>(L, stage, e + m + in, dn);
                extrapolate(L, y == 0 ? SOUTH : NORTH, dn, ev);
#pragma unroll
                for (int i = 0; i < 9; ++i) {
                    const float v = to_store<T>(L, i, ev[i]);
                    if (m == 0) dk[i].x = v; else dk[i].y = v;
                }
            }
        }

        // the segment's last reads of the stage are done: recycle it for the
        // warp's next segment
        if (pass == npass - 1) {
            __syncwarp();
            if (has_next) {
                fence_proxy_async_smem();
                const int ys = streamed_row<EDGES>(Ln, ny2);
                issue_segment<T>(srcn, Ln, ys, nx2, stage, ring.bar, lane);
                wv = wrap_load<T>(srcn, Ln, ys, nx2, lane);
                ring.pending = true;
            }
        }

        // ---- solid fraction (Eq. 14), owner and particle velocity per node:
        // max over the tile's candidates, lowest particle id on ties
        float phi[2] = {0.f, 0.f}, rxn[2] = {0.f, 0.f}, ryn[2] = {0.f, 0.f};
        int best[2] = {-1, -1};
        // (cands is warp-uniform; a segment no particle reaches skips all of it)
        for (unsigned left = cands; left; left &= left - 1) {
            const int c = __ffs(left) - 1;
            const float4 ra = crec[c], rb = crec[MAXC + c];
            const float R = rb.x + ph.cut;
            float dy = ((float)(y - ty0) - ra.z) - ra.w;
            // short periodic axes: the stored image may lie several periods away
            // (it is the one nearest the tile centre), so reduce by the nearest
            // multiple of the period (exact: an integer multiple of an integer)
            int ky = 0;                                     // PS: periods removed, for the table index
            if (L.wrap_y) {
                const float k = rintf(dy * __frcp_rn((float)L.ny));
                dy = fmaf(-(float)L.ny, k, dy);
                ky = (int)k;
            }
            const float h2 = fmaf(-dy, dy, R * R);
            if (h2 < 0.f) continue;                         // this row misses the disc tail
            const float dx0 = ((float)e - ra.x) - ra.y;
            if (!L.wrap_x) {
                // the pair spans [dx0, dx0 + 1]
                const float lo = dx0 > 0.f ? dx0 : (dx0 + 1.0f < 0.f ? -(dx0 + 1.0f) : 0.f);
                if (lo * lo > h2) continue;
            }
            const int id = cid[c];
            if constexpr (PS) {
                // covered cell fraction (B = eps_s, Eq. 8): 1 once every corner is
                // inside, else the particle's table entry for the cell.  Both
                // nodes' entries are fetched before either is used.  The
                // centre's whole-cell offsets come packed in the record.
                const int fpk = __float_as_int(crec[2 * MAXC + c].w);
                const int K = ph.ck, S = 2 * K + 1;
                const float *tab = A.B.cover + (long long)id * S * S;
                const int iy = (y - ty0) - (int)(short)((unsigned)fpk >> 16) - L.ny * ky + K;
                float pcq[2];
                float2 dxq = make_float2(dx0, dx0 + 1.0f);
                int kxq[2] = {0, 0};
                if (L.wrap_x) {
#pragma unroll
                    for (int m = 0; m < 2; ++m) {
                        const float k = rintf(slot(dxq, m) * __frcp_rn((float)L.nx));
                        slot(dxq, m) = fmaf(-(float)L.nx, k, slot(dxq, m));
                        kxq[m] = (int)k;
                    }
                }
                float2 d2q = fma2(dxq, dxq, f2(dy * dy)), lq = sub2(f2(rb.x), sqrt2(d2q));
#pragma unroll
                for (int m = 0; m < 2; ++m) {
                    const int kx = kxq[m];
                    const float d2 = slot(d2q, m), l = slot(lq, m);
                    const int ix = e + m - (int)(short)(fpk & 0xffff) - L.nx * kx + K;
                    const bool inside = d2 <= R * R && l >= -ph.cut;
                    const bool look = inside && l < ph.cut && (unsigned)ix < (unsigned)S && (unsigned)iy < (unsigned)S;
                    pcq[m] = look ? __ldcg(tab + iy * S + ix) : (inside && l >= ph.cut ? 1.0f : 0.f);
                }
#pragma unroll
                for (int m = 0; m < 2; ++m) {
                    const float pc = pcq[m];
                    if (!(pc > 0.f)) continue;
                    if (pc > phi[m] || (pc == phi[m] && id < cid[best[m]])) {
                        phi[m] = pc; best[m] = c; rxn[m] = slot(dxq, m); ryn[m] = dy;
                    }
                }
            } else {
                float2 dx = make_float2(dx0, dx0 + 1.0f);
                if (L.wrap_x) {
                    dx.x = fmaf(-(float)L.nx, rintf(dx.x * __frcp_rn((float)L.nx)), dx.x);
                    dx.y = fmaf(-(float)L.nx, rintf(dx.y * __frcp_rn((float)L.nx)), dx.y);
                }
                const float2 d2 = fma2(dx, dx, f2(dy * dy));
                const float2 l = sub2(f2(rb.x), sqrt2(d2));
                // (1 + tanh(2l/eps)) / 2 == 1 / (1 + exp(-4l/eps)) == 1 / (1 + 2^(phi_k2 l)),
                // with the hardware's base-2 exponential and reciprocal: the
                // rounding of the argument phi_k2 l (|.| <= 23 inside the tail,
                // a relative error of at most 23 * 2^-24 in the power) bounds
                // the error either way, and both instructions add about an ulp.
                // (Beyond the tail the value is not used.)
                const float2 a = mul2(f2(ph.phi_k2), l);
                const float2 den = add2(f2(1.0f), make_float2(ex2_approx(a.x), ex2_approx(a.y)));
                const float pcs[2] = {rcp_approx(den.x), rcp_approx(den.y)};
                const bool in[2] = {d2.x <= R * R && l.x >= -ph.cut, d2.y <= R * R && l.y >= -ph.cut};
#pragma unroll
                for (int m = 0; m < 2; ++m) {
                    const float pc = in[m] ? pcs[m] : 0.f;
                    if (pc > phi[m] || (pc == phi[m] && pc > 0.f && id < cid[best[m]])) {
                        phi[m] = pc; best[m] = c; rxn[m] = slot(dx, m); ryn[m] = dy;
                    }
                }
            }
        }

        // warps with no node inside any particle's phi tail collide without the force term
        const bool coupled = cands && __any_sync(0xffffffffu, max(best[0], best[1]) >= 0);
        const bool act_a = x < L.nx, act_b = x + 1 < L.nx;

        // ---- moments (Eq. 5, Eq. 16): of the stored values, then physical
        const float2 ms = add2(add2(add2(add2(dk[0], dk[1]), add2(dk[2], dk[3])),
                                    add2(add2(dk[4], dk[5]), add2(dk[6], dk[7]))), dk[8]);
        const float2 jxs = add2(add2(sub2(dk[1], dk[3]), sub2(dk[5], dk[6])), sub2(dk[8], dk[7]));
        const float2 jys = sub2(add2(sub2(dk[2], dk[4]), add2(dk[5], dk[6])), add2(dk[7], dk[8]));
        float2 drho = ms, jx = jxs, jy = jys;
        if constexpr (!std::is_same<T, float>::value) {
            const float2 q = f2(L.ref_q);
            drho = fma2(q, ms, f2(L.ref_m[0]));
            jx = fma2(q, jxs, f2(L.ref_m[1]));
            jy = fma2(q, jys, f2(L.ref_m[2]));
        }
        const float2 rho = add2(f2(1.0f), drho);
        // u* (Eq. 16); a correctly rounded reciprocal (a biased one would
        // bias u* the same way on every node and step)
        const float2 inv = recip2(rho);
        const float2 ua = mul2(jx, inv), va = mul2(jy, inv);
        if (MODE == MODE_STEP) {
            // unstable: rho <= 0 or not finite (a non-finite population makes
            // rho non-finite); as unsigned, bits(rho) - 1 exceeds the largest
            // finite float's bits - 1 exactly then
            badmax = max(badmax, act_a ? __float_as_uint(rho.x) - 1u : 0u);
            badmax = max(badmax, act_b ? __float_as_uint(rho.y) - 1u : 0u);
        }

        if (!coupled) {
            if (MODE == MODE_FIELDS) {
                const long long o = (long long)y * L.nx + x;
                if (act_a) {
                    if (fo.rho) fo.rho[o] = rho.x;
                    if (fo.ux) fo.ux[o] = ua.x;
                    if (fo.uy) fo.uy[o] = va.x;
                    if (fo.phi) fo.phi[o] = 0.f;
                }
                if (act_b) {
                    if (fo.rho) fo.rho[o + 1] = rho.y;
                    if (fo.ux) fo.ux[o + 1] = ua.y;
                    if (fo.uy) fo.uy[o + 1] = va.y;
                    if (fo.phi) fo.phi[o + 1] = 0.f;
                }
                continue;
            }
            collide_plain2<T>(dk, L, ph.omega, ms, jxs, jys, jx, jy, ua, va);
        } else {
            // u_s - u* from the particle velocity carried as FP32 hi + lo:
            // u_s = U + omega x r with r the node's offset from the centre
            float du[2] = {0.f, 0.f}, dv[2] = {0.f, 0.f};
            const float uas[2] = {ua.x, ua.y}, vas[2] = {va.x, va.y};
#pragma unroll
            for (int m = 0; m < 2; ++m) {
                const int b = best[m];
                if (b >= 0) {
                    const float4 rb = crec[MAXC + b], rl = crec[2 * MAXC + b];
                    du[m] = fmaf(-rb.w, ryn[m], rb.y - uas[m]) + fmaf(-rl.z, ryn[m], rl.x);
                    dv[m] = fmaf(rb.w, rxn[m], rb.z - vas[m]) + fmaf(rl.z, rxn[m], rl.y);
                }
            }
            const float2 dux = make_float2(du[0], du[1]), duy = make_float2(dv[0], dv[1]);
            const float2 usx = add2(ua, dux), usy = add2(va, duy);
            const float2 phq = make_float2(phi[0], phi[1]);
            // ---- corrected velocity (Eq. 17)
            // (PS-LBM: f^eq takes the fluid velocity u*, there is no correction)
            const float2 hph = mul2(f2(PS ? 0.0f : 0.5f), phq);
            const float2 ux = fma2(hph, dux, ua), uy = fma2(hph, duy, va);

            if (MODE == MODE_FIELDS) {
                const long long o = (long long)y * L.nx + x;
                if (act_a) {
                    if (fo.rho) fo.rho[o] = rho.x;
                    if (fo.ux) fo.ux[o] = ux.x;
                    if (fo.uy) fo.uy[o] = uy.x;
                    if (fo.phi) fo.phi[o] = phq.x;
                }
                if (act_b) {
                    if (fo.rho) fo.rho[o + 1] = rho.y;
                    if (fo.ux) fo.ux[o + 1] = ux.y;
                    if (fo.uy) fo.uy[o + 1] = uy.y;
                    if (fo.phi) fo.phi[o + 1] = phq.y;
                }
                continue;
            }
            const float2 prho = mul2(rho, phq);
            collide2<T>(dk, L, ph.omega, ms, jxs, jys, rho, ux, uy, mul2(f2(ph.kf), prho), prho, dux, duy, usx, usy,
                        ua, va);

            // ---- Eqs. 18-19 per node, by the closed form sum_i F_i c_i = kf rho (u_s - u*),
            // summed per candidate over the pass (the lane's two nodes, then a
            // fixed shuffle tree) and added to that candidate's lane
            const int own_a = act_a ? best[0] : -1, own_b = act_b ? best[1] : -1;
            const float sa = -prho.x * ph.kforce, sb = -prho.y * ph.kforce;
            const float gax = sa * du[0], gay = sa * dv[0], gbx = sb * du[1], gby = sb * dv[1];
            const float ta = fmaf(rxn[0], gay, -(ryn[0] * gax)), tb = fmaf(rxn[1], gby, -(ryn[1] * gbx));
            for (unsigned left = cands; left; left &= left - 1) {
                const int c = __ffs(left) - 1;
                if (!__any_sync(0xffffffffu, own_a == c || own_b == c)) continue;
                float v0 = 0.f, v1 = 0.f, v2 = 0.f;
                if (own_a == c) { v0 = gax; v1 = gay; v2 = ta; }
                if (own_b == c) { v0 += gbx; v1 += gby; v2 += tb; }
                // three sums over 32 lanes in 6 shuffles: at the tree's first
                // two levels the lanes part with a component each (as in
                // hydro_sums), so that lanes 0, 8 and 16 end with x, y and the
                // torque.  (One tree per component took 15.)
                const bool up = lane & 16, odd = lane & 8;
                const float r0 = __shfl_xor_sync(0xffffffffu, up ? v0 : v2, 16), r1 = __shfl_xor_sync(0xffffffffu, v1, 16);
                const float b0 = (up ? v2 : v0) + r0, b1 = v1 + r1;
                float g = (odd ? b1 : b0) + __shfl_xor_sync(0xffffffffu, odd ? b0 : b1, 8);
#pragma unroll
                for (int o = 4; o > 0; o >>= 1) g += __shfl_xor_sync(0xffffffffu, g, o);
                if ((lane & 7) == 0 && lane < 24) reinterpret_cast<float *>(crec + NREC * MAXC + c)[lane >> 3] += g;
            }
        }

        // ---- store the collided pair: one contiguous run per plane and pass
        T *base = dst + (long long)y * L.row + x;
        if (act_b) {
#pragma unroll
            for (int i = 0; i < 9; ++i) Storage<T>::store2(base + i * L.plane, dk[i]);
        } else if (act_a) {
#pragma unroll
            for (int i = 0; i < 9; ++i) Storage<T>::store1(base + i * L.plane, dk[i].x);
        }
    }

    if (MODE == MODE_FIELDS) return true;
    if (__any_sync(0xffffffffu, badmax > 0x7f7ffffeu) && lane == 0) atomicOr(A.err, ERR_UNSTABLE);
    // ---- this row segment's force / torque per candidate (zero where no node is owned)
    if (HALVES) meet_partner();
    else __syncwarp();
    if (HALVES && half == 1) return true;
    if (cands >> lane & 1u) {
        float4 sg = crec[NREC * MAXC + lane];
        if (HALVES) {
            // the partner's, the second pass's, added as one warp adds them
            const float4 s2 = crec[(NREC + 1) * MAXC + NREC * MAXC + lane];
            sg.x += s2.x; sg.y += s2.y; sg.z += s2.z;
        }
        const int id = cid[lane];
        const long long entry = A.B.by_slot ? (long long)tile * MAXC + lane : (long long)id * MAXT + __float_as_int(sg.w);
        float4 *out = A.partial + entry * TILE_H + (y - ty0);
        if (FUSED) {
            store_partial(out, sg.x, sg.y, sg.z, tag);
            if (count) count_done(B.done + id);
        } else {
            *out = make_float4(sg.x, sg.y, sg.z, 0.f);
        }
    }
    return true;
}

// Shared-memory carve-up of the sweep kernels.
template <typename T, int W>
struct SweepSmem {
    T *stage;
    float4 *crec;
    int *cid;
    uint64_t *bar;
    __device__ __forceinline__ SweepSmem(unsigned char *raw, int warp) {
        constexpr size_t STAGE_BYTES = (size_t)W * stage_elems<T>() * sizeof(T);
        constexpr size_t REC_BYTES = (size_t)W * (NREC + 1) * MAXC * sizeof(float4);
        constexpr size_t ID_BYTES = (size_t)W * MAXC * sizeof(int);
        stage = reinterpret_cast<T *>(raw) + (size_t)warp * stage_elems<T>();
        crec = reinterpret_cast<float4 *>(raw + STAGE_BYTES) + (size_t)warp * (NREC + 1) * MAXC;
        cid = reinterpret_cast<int *>(raw + STAGE_BYTES + REC_BYTES) + warp * MAXC;
        bar = reinterpret_cast<uint64_t *>(raw + STAGE_BYTES + REC_BYTES + ID_BYTES) + warp;
    }
};

// Resident warps per SM the sweep kernels are compiled for: W warps per block
// and sm_warps / W blocks per SM (registers capped at 96 per thread in FP32
// storage for W = 2 and 4, at 80 in 16-bit storage; W = 8 holds two blocks in
// FP32, 16 warps).
template <typename T> constexpr int sm_warps() { return sizeof(T) == 4 ? 20 : 24; }

// Row of item `item` (row-major over rows of ntx segments) without a
// division: inv = floor(2^32 / ntx) + 1 overestimates the quotient by less
// than item / 2^32 < 1, so one correction makes it exact.
__device__ __forceinline__ int row_of(unsigned item, unsigned inv, int ntx) {
    if (ntx == 1) return (int)item;
    unsigned q = __umulhi(item, inv);
    if (q * (unsigned)ntx > item) --q;
    return (int)q;
}

// The sweep over one lattice without the particle update (a strip's step, the
// static step, a step of a small lattice without particles, and the fields).  Persistent: warps take row segments
// round-robin (neighbouring warps on neighbouring segments); each warp keeps
// its next segment staged ahead.  W warps per block.
template <typename T, int MODE, bool EDGES, bool PS, int W>
__global__ void __launch_bounds__(W * 32, 20 / W)
sweep_kernel(const __grid_constant__ SweepArgs<T> one, const __grid_constant__ FieldsOut fo)
{
    extern __shared__ __align__(128) unsigned char smem_raw[];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    SweepSmem<T, W> sm(smem_raw, warp);
    Ring ring{sm.bar, 0u, false};
    if (lane == 0) {
        mbar_init(ring.bar, 1);
        mbar_fence_init();
    }
    __syncwarp();
    // Launched while the step before still runs (sweep_variant, `chained`): wait
    // for its end here, and let the step after come as this one's blocks leave.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const Lattice &L = one.L;
    const T *src = one.buf[one.cur];
    T *dst = one.buf[one.cur ^ 1];
    const Bins bins = bins_at(one.B, one.cur, one.clock ? __ldcg(&one.clock->rot) : one.cur);
    // the next step's bins start empty (nothing reads them during this sweep)
    if (MODE == MODE_STEP && one.np > 0) {
        int *clear = one.B.count + (long long)(one.cur ^ 1) * one.B.tiles;
        for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < L.ntx * L.nty; t += gridDim.x * blockDim.x) clear[t] = 0;
    }
    if (MODE == MODE_STEP && one.clock && blockIdx.x == 0 && threadIdx.x == 0) one.clock->tag += 1;
    const int nitems = L.ny * L.ntx;
    const int gw = blockIdx.x * W + warp, nw = gridDim.x * W;
    T wv = T();         // the staged segment's periodic-edge value (wrap_load)
    // (from the end where the next step would: see SweepArgs::turn)
    auto seek = [&](int k, int &sy, int &sx) {
        const int item = one.turn && one.cur && k < nitems ? nitems - 1 - k : k;
        sy = row_of(item, one.ntx_inv, L.ntx);
        sx = item - sy * L.ntx;
    };
    int y, tx;
    seek(gw, y, tx);
    if (gw < nitems) {
        issue_segment<T>(src, L, streamed_row<EDGES>(L, y), tx, sm.stage, ring.bar, lane);
        wv = wrap_load<T>(src, L, streamed_row<EDGES>(L, y), tx, lane);
        ring.pending = true;
    }
    bool timed_out = false;
    for (int item = gw; item < nitems; item += nw) {
        const int nxt = item + nw;
        const bool has_next = nxt < nitems;
        int ny2, nx2;
        seek(nxt, ny2, nx2);
        if (!sweep_segment<T, MODE, EDGES, PS, false>(one, src, dst, bins, y, tx, sm.stage, ring, has_next, src, L, ny2,
                                                      nx2, sm.crec, sm.cid, wv, 0u, false, fo, lane)) {
            timed_out = true;
            break;
        }
        y = ny2;
        tx = nx2;
    }
    if (timed_out) {
        if (lane == 0) atomicOr(one.err, ERR_TIMEOUT);
        // let the copies this warp still has in flight land before the block
        // releases its shared memory (the wait bounded again)
        if (ring.pending) mbar_wait_bounded(ring.bar, ring.parity);
    }
}

// ------------------------------------------------------------ particles
struct BodyParams {
    int np;
    double gx, gy, rho_f;
    double eps_p, eps_p2, eps_w, eps_w2, xi;
    double len[2];              // nx, ny
    float xi_f;
};

// Map k in [0, total) of a tile-range set to its tile index, ranges in order.
__device__ __forceinline__ int range_at(const AxisTiles &a, int k) {
    const int n0 = a.hi[0] - a.lo[0] + 1;
    return k < n0 ? a.lo[0] + k : a.lo[1] + (k - n0);
}

__device__ __forceinline__ int range_len(const AxisTiles &a) {
    int n = 0;
    for (int r = 0; r < a.n; ++r) n += a.hi[r] - a.lo[r] + 1;
    return n;
}

// Everything one lattice's particle update needs, whatever the step.
struct PartArgs {
    Lattice L;
    Physics ph;
    Particles P;
    BodyParams bp;
    BinSet B;
    float4 *partial;
    double *force, *fcol;
    double *fsum;               // nullable: running sum of (Fx, Fy, T) over integrating steps
    int *err;
    StepClock *clock = nullptr;       // (null: see StepClock)
    int track = -1;             // moving frame: tracked particle, -1 (the default) when off
    double track_x = 0.0;       // its reference x
    long long *frame_off = nullptr;   // columns the frame has moved
    // A strip of the lattice (L is the whole lattice): bins hold the tile rows
    // [ty_lo, ty_hi) only, local tile index (ty - ty_lo) * ntx + tx.
    int ty_lo = 0, ty_hi = 1 << 30;
    double *fpart = nullptr;    // a strip's sums (5 per particle: Fx, Fy, T, repulsion x, y)
};

// v wrapped into [0, n) on a periodic axis: fmod(v, n), plus n when it is
// negative.  A position moves by less than a period per step, so within
// (-n, 2n) one subtraction or addition of n gives exactly that result (the
// difference is representable); fmod takes anything farther, and NaN.
__host__ __device__ inline double wrap_period(double v, double n) {
    if (v >= 0.0 && v < n) return v;
    if (v >= n && v < 2.0 * n) return v - n;
    if (v < 0.0 && v > -n) return v + n;
    const double w = fmod(v, n);
    return w < 0.0 ? w + n : w;
}

// Moving computational domain (Sec. 3.5): the frame's move at the end of a
// step, in columns, from the tracked particle's x at the start of that step
// (minimum image on a periodic x axis): +1 once it is one lattice unit or
// more ahead of the reference, -1 once one or more behind.
__host__ __device__ inline int frame_move(double xt, double xref, int nx, int per_x) {
    double d = xt - xref;
    if (per_x) {
        while (d >= 0.5 * nx) d -= nx;
        while (d < -0.5 * nx) d += nx;
    }
    return d >= 1.0 ? 1 : (d <= -1.0 ? -1 : 0);
}

// The particle update of one step, by one warp per particle, in three parts:
//   contact  -- Wan-Turek repulsion (Eqs. 28-29) from the other particles
//               (lanes stride over the particle's tiles) and from mirror
//               images across the walls.  It reads only the step's starting
//               positions, so it runs at the start of a step, off the chain
//               that the forces are on;
//   sums     -- hydrodynamic force and torque (Eqs. 18-19): the row-segment
//               partials, summed in FP64 in a fixed order (lanes take fixed
//               (tile, row) entries, then a fixed shuffle tree);
//   advance  -- symplectic Euler of Eqs. 22-24 (dt = 1), then binning of the
//               particle into every tile its phi tail reaches.
// Everything a step changes is read from L2 (__ldcg): in a launch over several
// steps another SM wrote it, and the L1 is not coherent.

struct Repulsion {
    double x, y;
};

// Could particle p be within Eq. 28's range of another one?  Each lane takes
// one (tile, slot) of the particle's first eight tiles and first four taken slots
// and compares the two records there (FP32, relative to the tile, with a
// margin far above their rounding), so that the answer takes two dependent
// loads; more tiles or slots, or a periodic axis too short for one image per
// tile, answer yes.
__device__ __forceinline__ bool maybe_near(const PartArgs &A, int p, const Bins &B, int lane) {
    const int nk = __ldcg(B.npslot + p);
    const int k = lane >> 2, sl = lane & 3;
    const int t = listed_tile(__ldcg(B.pslot + (long long)p * MAXT + k));       // (entries past nk: stale, or never written)
    bool far = nk <= 8 && !A.L.wrap_x && !A.L.wrap_y;
    float4 ra = make_float4(0.f, 0.f, 0.f, 0.f), rb = ra;
    int id = -1, n = 0;
    if (k < nk && t >= 0) {
        unsigned m = (unsigned)__ldcg(B.count + t);
        int s = sl;
        if (masked_bins(A.bp.np)) {
            n = __popc(m);
            for (int i = 0; i < sl; ++i) m &= m - 1;
            s = m ? __ffs(m) - 1 : 0;
        } else {
            n = (int)m;
        }
        const long long q = (long long)t * MAXC + s;
        id = __ldcg(&B.ids[q].x);
        ra = __ldcg(B.rec + NREC * q);
        rb = __ldcg(B.rec + NREC * q + 1);
    } else if (k < nk) {
        far = false;
    }
    far = far && n <= 4;
    if (sl >= n) id = -1;
    // the particle's own record among the tile's four
    const unsigned mine = __ballot_sync(0xffffffffu, id == p) >> (lane & 28) & 15u;
    const int src = (lane & 28) + (mine ? __ffs(mine) - 1 : 0);
    const float dx = (ra.x - __shfl_sync(0xffffffffu, ra.x, src)) + (ra.y - __shfl_sync(0xffffffffu, ra.y, src));
    const float dy = (ra.z - __shfl_sync(0xffffffffu, ra.z, src)) + (ra.w - __shfl_sync(0xffffffffu, ra.w, src));
    const float lim = rb.x + __shfl_sync(0xffffffffu, rb.x, src) + A.bp.xi_f + 0.05f;
    if (id >= 0 && id != p && !(dx * dx + dy * dy > lim * lim)) far = false;
    if (n > 0 && !mine) far = false;
    return !__all_sync(0xffffffffu, far);
}

// The pairs (Eq. 28), summed over the warp.
__device__ __forceinline__ Repulsion pair_repulsion(const PartArgs &A, int p, int cur, const Bins &B, int lane) {
    const Lattice &L = A.L;
    const Particles &P = A.P;
    const BodyParams &bp = A.bp;
    const double *xin = cur ? P.x[1] : P.x[0], *yin = cur ? P.y[1] : P.y[0];
    const float *xfin = cur ? P.xf[1] : P.xf[0], *yfin = cur ? P.yf[1] : P.yf[0];
    double cx = 0.0, cy = 0.0;
    if (bp.np > 1 && maybe_near(A, p, B, lane)) {
        const double X = __ldcg(xin + p), Y = __ldcg(yin + p), r = __ldcg(P.r + p);
        const float xf = __ldcg(xfin + p), yf = __ldcg(yfin + p), rf = __ldcg(P.rf + p);
        const int nk = __ldcg(B.npslot + p);
        // A pair within r_i + r_j + xi shares the tile holding the middle of
        // the gap between the surfaces (that point lies inside both binning
        // reaches), so each lane takes some of this particle's tiles and
        // counts a pair only in that tile; within a tile the pairs are added
        // in increasing partner id.
        for (int k = lane; k < nk; k += 32) {
            const int t = listed_tile(__ldcg(B.pslot + (long long)p * MAXT + k));
            if (t < 0) continue;
            uint32_t contact = 0;
            for (unsigned taken = slot_mask(__ldcg(B.count + t), bp.np); taken; taken &= taken - 1) {
                const int sl = __ffs(taken) - 1;
                const int j = __ldcg(&B.ids[(long long)t * MAXC + sl].x);
                if (j == p) continue;
                float dxf = xf - __ldcg(xfin + j), dyf = yf - __ldcg(yfin + j);
                if (L.per_x) { if (dxf >= 0.5f * L.nx) dxf -= L.nx; else if (dxf < -0.5f * L.nx) dxf += L.nx; }
                if (L.per_y) { if (dyf >= 0.5f * L.ny) dyf -= L.ny; else if (dyf < -0.5f * L.ny) dyf += L.ny; }
                const float lim = rf + __ldcg(P.rf + j) + bp.xi_f + 0.05f;
                if (dxf * dxf + dyf * dyf > lim * lim) continue;
                const double rj = __ldcg(P.r + j);
                double dx = X - __ldcg(xin + j), dy = Y - __ldcg(yin + j);
                if (L.per_x) { while (dx >= 0.5 * L.nx) dx -= L.nx; while (dx < -0.5 * L.nx) dx += L.nx; }
                if (L.per_y) { while (dy >= 0.5 * L.ny) dy -= L.ny; while (dy < -0.5 * L.ny) dy += L.ny; }
                // the middle of the gap between the two surfaces, at distance
                // (d + r - r_j) / 2 from this centre toward the partner
                const double dd = sqrt(dx * dx + dy * dy);
                const double f = dd > 0.0 ? 0.5 * (dd + r - rj) / dd : 0.0;
                double mx = X - f * dx, my = Y - f * dy;
                if (L.per_x) mx = wrap_period(mx, (double)L.nx);
                if (L.per_y) my = wrap_period(my, (double)L.ny);
                int mxi = (int)floor(mx), myi = (int)floor(my);
                mxi = mxi < 0 ? 0 : (mxi > L.nx - 1 ? L.nx - 1 : mxi);
                myi = myi < 0 ? 0 : (myi > L.ny - 1 ? L.ny - 1 : myi);
                if ((myi / TILE_H) * L.ntx + mxi / TILE_W == t + A.ty_lo * L.ntx) contact |= 1u << sl;
            }
            while (contact) {                         // increasing partner id
                int sel = -1, jmin = 0x7fffffff;
                for (uint32_t m = contact; m; m &= m - 1) {
                    const int sl = __ffs(m) - 1, j = __ldcg(&B.ids[(long long)t * MAXC + sl].x);
                    if (j < jmin) { jmin = j; sel = sl; }
                }
                contact &= ~(1u << sel);
                double dx = X - __ldcg(xin + jmin), dy = Y - __ldcg(yin + jmin);
                if (L.per_x) { while (dx >= 0.5 * L.nx) dx -= L.nx; while (dx < -0.5 * L.nx) dx += L.nx; }
                if (L.per_y) { while (dy >= 0.5 * L.ny) dy -= L.ny; while (dy < -0.5 * L.ny) dy += L.ny; }
                const double d = sqrt(dx * dx + dy * dy), rr = r + __ldcg(P.r + jmin);
                double sc = 0.0;
                if (d <= rr) sc = (rr - d) / bp.eps_p2;
                else if (d <= rr + bp.xi) sc = (rr + bp.xi - d) * (rr + bp.xi - d) / bp.eps_p;
                cx += sc * dx;
                cy += sc * dy;
            }
        }
        // (zero unless some lane found a contact: reduced only when one did)
        if (__any_sync(0xffffffffu, cx != 0.0 || cy != 0.0)) {
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) {
                cx += __shfl_xor_sync(0xffffffffu, cx, o);
                cy += __shfl_xor_sync(0xffffffffu, cy, o);
            }
        }
    }
    return Repulsion{cx, cy};
}

// The walls (Eq. 29): the mirror image across each non-periodic wall, added
// to the pairs' sum wall by wall.
__device__ __forceinline__ void wall_repulsion(const PartArgs &A, int p, int cur, Repulsion &c) {
    const Lattice &L = A.L;
    const BodyParams &bp = A.bp;
    if (L.per_x && L.per_y) return;
    {
        // FP32, with a margin above its rounding: out of every wall's range?
        const float x = __ldcg((cur ? A.P.xf[1] : A.P.xf[0]) + p), y = __ldcg((cur ? A.P.yf[1] : A.P.yf[0]) + p);
        const float nx1 = (float)(L.nx - 1), ny1 = (float)(L.ny - 1);
        const float lim = __ldcg(A.P.rf + p) + 0.5f * bp.xi_f + 0.25f + 1e-6f * fmaxf(nx1, ny1);
        if ((L.per_x || (x > lim && nx1 - x > lim)) && (L.per_y || (y > lim && ny1 - y > lim))) return;
    }
    const double X = __ldcg((cur ? A.P.x[1] : A.P.x[0]) + p), Y = __ldcg((cur ? A.P.y[1] : A.P.y[0]) + p);
    const double r = __ldcg(A.P.r + p);
    for (int w = 0; w < 4; ++w) {
        if (L.side_kind[w] == SIDE_PERIODIC) continue;
        double ix = X, iy = Y;
        if (w == WEST) ix = -X;
        if (w == EAST) ix = 2.0 * (L.nx - 1) - X;
        if (w == SOUTH) iy = -Y;
        if (w == NORTH) iy = 2.0 * (L.ny - 1) - Y;
        const double dx = X - ix, dy = Y - iy;
        const double d = sqrt(dx * dx + dy * dy), rr = 2.0 * r;
        double sc = 0.0;
        if (d <= rr) sc = (rr - d) / bp.eps_w2;
        else if (d <= rr + bp.xi) sc = (rr + bp.xi - d) * (rr + bp.xi - d) / bp.eps_w;
        c.x += sc * dx;
        c.y += sc * dy;
    }
}

// An FP32 value as FP64 (exact).  Normal values and zeros on the integer
// pipe: an FP64-pipe instruction takes a warp as long as dozens of others.
__device__ __forceinline__ double widen(float v) {
    const uint32_t u = __float_as_uint(v), e = (u >> 23) & 255u;
    if (e - 1u < 254u)
        return __hiloint2double((int)((u & 0x80000000u) | (((u & 0x7fffffffu) >> 3) + 0x38000000u)), (int)(u << 29));
    if ((u << 1) == 0u) return __hiloint2double((int)u, 0);
    return (double)v;
}

// The particle update's scalar part runs with one component per group of
// eight lanes (0: x, 1: y, 2: rotation, 3: idle), so that an FP64 instruction
// serves all three.
__device__ __forceinline__ int component(int lane) { return lane >> 3; }

// Particle p's force and torque (Eqs. 18-19), each in its component's lanes:
// lane l adds entries e = l, l + 32, ... (tile e / TILE_H of the particle's
// list, row e % TILE_H) in that order, then a fixed shuffle tree, in which the
// lanes part with a component at each of its first two levels (the sums are
// those of three whole trees).  The partials lie per particle in that order
// (rows outside the lattice and tiles of another strip hold zeros), so the
// first loads need nothing but p.  TAGGED: each entry is read until it carries
// the step's tag; the wait is bounded, and sets *late when it gives up.
template <bool TAGGED>
__device__ __forceinline__ double hydro_sums(const PartArgs &A, int p, const Bins &B, unsigned tag, int lane, bool *late) {
    double fx = 0.0, fy = 0.0, tq = 0.0;
    if (A.B.by_slot) {
        // the same entries in the same order, found by the list's slots
        const int ne = __ldcg(B.npslot + p) * TILE_H;
        for (int e = lane; e < ne + lane; e += 32) {
            const unsigned w = e < ne ? (unsigned)__ldcg(B.pslot + (long long)p * MAXT + e / TILE_H) : ~0u;
            const bool has = w != ~0u && ((int)(w / MAXC) / A.L.ntx + A.ty_lo) * TILE_H + e % TILE_H < A.L.ny;
            const float4 *from = A.partial + (long long)w * TILE_H + e % TILE_H;
            float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
            if (has) v = load_partial(from);
            unsigned long long t0 = 0;
            while (TAGGED) {
                const bool miss = has && __float_as_uint(v.w) != tag;
                if (!__any_sync(0xffffffffu, miss)) break;
                const unsigned long long t = global_ns();
                if (t0 == 0) t0 = t;
                *late = __any_sync(0xffffffffu, t - t0 > WAIT_LIMIT_NS);
                if (*late) break;
                if (miss) v = load_partial(from);
            }
            if (e == lane) {
                fx = widen(v.x); fy = widen(v.y); tq = widen(v.z);
            } else {
                fx += widen(v.x); fy += widen(v.y); tq += widen(v.z);
            }
        }
    } else {
        constexpr int Q = 3;        // entries per lane held at once (and waited for together)
        const float4 *part = A.partial + (long long)p * (MAXT * TILE_H) + lane;
        float4 v[Q];
#pragma unroll
        for (int q = 0; q < Q; ++q) v[q] = load_partial(part + 32 * q);
        const int ne = __ldcg(B.npslot + p) * TILE_H - lane;        // entries from this lane's first on
        for (int base = 0; base < ne + lane; base += 32 * Q) {
            if (base > 0) {
#pragma unroll
                for (int q = 0; q < Q; ++q)
                    if (base + 32 * q < ne) v[q] = load_partial(part + base + 32 * q);
            }
            unsigned long long t0 = 0;
            while (TAGGED) {
                bool miss = false;
#pragma unroll
                for (int q = 0; q < Q; ++q)
                    if (base + 32 * q < ne && __float_as_uint(v[q].w) != tag) {
                        v[q] = load_partial(part + base + 32 * q);
                        miss = true;
                    }
                // (together: lanes that left on their own would sum on their own)
                if (!__any_sync(0xffffffffu, miss)) break;
                const unsigned long long t = global_ns();
                if (t0 == 0) t0 = t;
                *late = __any_sync(0xffffffffu, t - t0 > WAIT_LIMIT_NS);
                if (*late) break;
            }
#pragma unroll
            for (int q = 0; q < Q; ++q) {
                if (base + 32 * q >= ne) break;
                if (base + q == 0) {
                    fx = widen(v[q].x); fy = widen(v[q].y); tq = widen(v[q].z);
                } else {
                    fx += widen(v[q].x); fy += widen(v[q].y); tq += widen(v[q].z);
                }
            }
        }
    }
    const bool up = lane & 16, odd = lane & 8;
    const double r0 = __shfl_xor_sync(0xffffffffu, up ? fx : tq, 16), r1 = __shfl_xor_sync(0xffffffffu, fy, 16);
    const double b0 = (up ? tq : fx) + r0, b1 = fy + r1;
    double f = (odd ? b1 : b0) + __shfl_xor_sync(0xffffffffu, odd ? b0 : b1, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) f += __shfl_xor_sync(0xffffffffu, f, o);
    return f;
}

// What particle_advance reads of a particle, one component per lane group.
// Loaded in one go, before or together with the partials.
struct PartState {
    double pos, vel, inv, weight, reach;    // x / y / theta, its rate, 1/m or 1/I, weight, reach
    double sum;                             // running sum of the force (PartArgs::fsum)
    float rf;
    int fixed;
};

__device__ __forceinline__ PartState load_particle(const PartArgs &A, int p, int cur, int lane) {
    const Particles &P = A.P;
    const int c = component(lane);
    PartState s;
    s.pos = __ldcg((c == 0 ? (cur ? P.x[1] : P.x[0]) : (c == 1 ? (cur ? P.y[1] : P.y[0]) : P.theta)) + p);
    s.vel = __ldcg((c == 0 ? P.ux : (c == 1 ? P.uy : P.omega)) + p);
    s.inv = __ldcg((c < 2 ? P.im : P.iI) + p);
    s.weight = c < 2 ? __ldcg((c == 0 ? P.wx : P.wy) + p) : 0.0;
    s.reach = __ldcg(P.reach + p);
    s.sum = A.fsum && c < 3 ? __ldcg(A.fsum + 3 * (long long)p + c) : 0.0;
    s.rf = __ldcg(P.rf + p);
    s.fixed = __ldcg(P.fixed + p);
    return s;
}

// Rigid-body update of particle p (Eqs. 22-24) from the force f and the
// repulsion c of this lane's component, positions copy `nxt` written -- with
// integrate == false the particle stays where it is -- then its binning into
// every tile its reach covers (in a fixed order), with the record the sweep
// reads: the centre relative to the tile origin (minimum image about the tile
// centre) as FP32 hi + lo, radius and velocities.  `out`: the bins the next
// sweep reads; `shift`: the frame's move.
__device__ __forceinline__ void particle_advance(const PartArgs &A, int p, const PartState &st, int nxt, const Bins &out,
                                                 bool integrate, int shift, unsigned next_tag, double f, double c,
                                                 int lane) {
    const Lattice &L = A.L;
    const Particles &P = A.P;
    const int comp = component(lane);
    const bool periodic = comp == 0 ? L.per_x : (comp == 1 ? L.per_y : false);
    const double len = comp == 0 ? A.bp.len[0] : A.bp.len[1];
    double u = st.vel, n = st.pos;
    auto wrap = [&]() {
        // (as integers: non-negative and below len, the usual case)
        if (periodic && (unsigned long long)__double_as_longlong(n) >= (unsigned long long)__double_as_longlong(len))
            n = wrap_period(n, len);
    };
    if (integrate) {
        const bool lead = (lane & 7) == 0 && comp < 3;
        if (!st.fixed) {
            u += (f + c + st.weight) * st.inv;
            n += u;
            wrap();
            if (lead) (comp == 0 ? P.ux : (comp == 1 ? P.uy : P.omega))[p] = u;
        }
        if (shift && comp == 0) {
            // the frame moves with the tracked particle: every particle, fixed
            // ones included, shifts by the same whole number of columns
            n -= (double)shift;
            wrap();
        }
        if (lead) {
            A.force[3 * (long long)p + comp] = f;
            if (A.fsum) A.fsum[3 * (long long)p + comp] = st.sum + f;
            if (comp == 2 && !st.fixed) P.theta[p] = n;
        }
    }
    if ((lane & 7) == 0 && comp < 2) {
        (comp == 0 ? (nxt ? P.x[1] : P.x[0]) : (nxt ? P.y[1] : P.y[0]))[p] = n;
        (comp == 0 ? (nxt ? P.xf[1] : P.xf[0]) : (nxt ? P.yf[1] : P.yf[0]))[p] = (float)n;
    }
    // velocities as FP32 hi + lo: the sweep forms u_s - u*, a small difference
    const float uh = (float)u, ul = (float)(u - widen(uh));
    const float uxh = __shfl_sync(0xffffffffu, uh, 0), uyh = __shfl_sync(0xffffffffu, uh, 8);
    const float omh = __shfl_sync(0xffffffffu, uh, 16), uxl = __shfl_sync(0xffffffffu, ul, 0);
    const float uyl = __shfl_sync(0xffffffffu, ul, 8), oml = __shfl_sync(0xffffffffu, ul, 16);
    // the tiles along the lane's axis
    const AxisTiles at = axis_tiles(n, st.reach, comp == 0 ? L.nx : L.ny, comp == 0 ? TILE_W_LOG2 : TILE_H_LOG2,
                                    comp == 0 ? L.ntx : L.nty, comp == 0 ? L.per_x : L.per_y);
    AxisTiles ax, ay;
    ax.n = __shfl_sync(0xffffffffu, at.n, 0);
    ay.n = __shfl_sync(0xffffffffu, at.n, 8);
#pragma unroll
    for (int q = 0; q < 2; ++q) {
        if (q == 1 && ax.n < 2 && ay.n < 2) break;
        ax.lo[q] = __shfl_sync(0xffffffffu, at.lo[q], 0);
        ax.hi[q] = __shfl_sync(0xffffffffu, at.hi[q], 0);
        ay.lo[q] = __shfl_sync(0xffffffffu, at.lo[q], 8);
        ay.hi[q] = __shfl_sync(0xffffffffu, at.hi[q], 8);
    }
    const double nX = __shfl_sync(0xffffffffu, n, 0), nY = __shfl_sync(0xffffffffu, n, 8);
    const int NX = range_len(ax), NY = range_len(ay);
    int total = NX * NY;
    if (total > MAXT) {                      // ruled out at create; kept as a guard
        if (lane == 0) atomicOr(A.err, ERR_OVERFLOW);
        total = MAXT;
    }
    // binning: two lanes per tile, one for each axis of its record
    const bool axis = lane & 1;
    int need = 0;                            // partials the next update waits for
    for (int k0 = 0; k0 < total; k0 += 16) {
        const int k = k0 + (lane >> 1);
        const bool has = k < total;
        int ty = 0, tx = 0;
        if (has) {
            const int ky = NX == 1 ? k : (NX == 2 ? k >> 1 : k / NX);
            ty = range_at(ay, ky);
            tx = range_at(ax, k - ky * NX);
        }
        const bool local = has && ty >= A.ty_lo && ty < A.ty_hi;        // (else another strip's tile)
        const int t = (ty - A.ty_lo) * L.ntx + tx;
        int s = MAXC;
        if (masked_bins(A.bp.np)) {
            if (local && !axis) atomicOr(&out.count[t], (int)(1u << p));
            s = p;
        } else if (local && !axis) {
            s = atomicAdd(&out.count[t], 1);
        }
        // the centre along the lane's axis, while the count's answer is on its way
        double r = (axis ? nY : nX) - (double)(axis ? ty * TILE_H : tx * TILE_W);
        float rh = (float)r;
        if (axis ? L.per_y : L.per_x) {
            const float h = axis ? 0.5f * TILE_H : 0.5f * TILE_W;
            const int ln = axis ? L.ny : L.nx;
            if (!(fabsf(rh - h) < 0.5f * (float)ln - 1.0f - 1e-6f * (float)ln)) {     // (else certainly the nearest image)
                while (r - (double)h >= 0.5 * ln) r -= ln;
                while (r - (double)h < -0.5 * ln) r += ln;
                rh = (float)r;
            }
        }
        const float rl = (float)(r - widen(rh));
        // the centre's whole-cell offsets from the tile origin (the PS sweep's table index)
        const int cell = __double2int_rd(r), other = __shfl_xor_sync(0xffffffffu, cell, 1);
        s = __shfl_sync(0xffffffffu, s, lane & 30);
        const bool in = local && s < MAXC;
        if (local && !in && !axis) atomicOr(A.err, ERR_OVERFLOW);
        int rows = 0;
        if (in) {
            rows = L.ny - ty * TILE_H;
            rows = rows < TILE_H ? rows : TILE_H;
            const long long q = (long long)t * MAXC + s;
            float2 *rec = reinterpret_cast<float2 *>(out.rec + NREC * q);
            rec[axis] = make_float2(rh, rl);
            if (!axis) {
                out.ids[q] = make_int2(p, k);
                out.rec[NREC * q + 1] = make_float4(st.rf, uxh, uyh, omh);
            } else {
                out.rec[NREC * q + 2] =
                    make_float4(uxl, uyl, oml, __int_as_float((other & 0xffff) | (int)((unsigned)cell << 16)));
            }
        }
        if (has && !axis) {
            out.pslot[(long long)p * MAXT + k] = in ? (int)((unsigned)t * MAXC + s) : -1;
            need += rows;
            // (this particle's partials of the step are summed: the entries no
            // sweep will write hold zero; an upload may replace a binning for
            // the same step, so it also takes that binning's tags off the others)
            for (int q = 0; !integrate && !A.B.by_slot && q < rows; ++q)
                store_partial(A.partial + ((long long)p * MAXT + k) * TILE_H + q, 0.f, 0.f, 0.f, next_tag - 1);
            for (int q = A.B.by_slot ? TILE_H : rows; q < TILE_H; ++q)
                store_partial(A.partial + ((long long)p * MAXT + k) * TILE_H + q, 0.f, 0.f, 0.f, next_tag);
        }
    }
    need = __reduce_add_sync(0xffffffffu, need);
    if (lane == 0) {
        out.npslot[p] = total;
        out.done[p] = -need;
    }
}

// New particles (an upload, or where they stand as a context starts), one warp
// per particle: forms 1/m, 1/I, weight and reach and bins the particle where it
// is.  `in`: the uploaded values in pinned host memory (x, y, r, ux, uy, omega,
// theta, rho_s, np doubles each, then np ints `fixed`), read in place; null:
// they are in device memory already.
// With a clock, one launch does it all: the particles go into the tile counts
// that a step would have added to (zero by then), the counts after them are
// zeroed in their place, and the last block out moves the clock on to the new
// ones.  (Four copies, a pass that cleared the counts and the binning took the
// coupled 512^2 step 64 us, this 48.)  Without a clock the caller has zeroed
// the counts of parity `cur`.
constexpr int PART_WARPS = 8;

static __global__ void __launch_bounds__(PART_WARPS * 32)
bin_particles_kernel(const __grid_constant__ PartArgs A, int cur, const double *__restrict__ in, unsigned *left) {
    const int lane = threadIdx.x & 31, p = blockIdx.x * PART_WARPS + (threadIdx.x >> 5), np = A.bp.np;
    const int rot = A.clock ? rot3(__ldcg(&A.clock->rot) + 1) : cur;
    if (A.clock) {
        int *zero = A.B.count + (long long)rot3(rot + 1) * A.B.tiles;
        for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < A.B.tiles; t += gridDim.x * blockDim.x) zero[t] = 0;
    }
    if (p < np) {
        const Particles &P = A.P;
        if (in) {
            // r .. rho_s lie one after another
            if (lane < 8) (lane == 0 ? P.x[cur] : (lane == 1 ? P.y[cur] : P.r + (lane - 2) * (long long)np))[p] = in[lane * (long long)np + p];
            if (lane == 8) P.fixed[p] = reinterpret_cast<const int *>(in + 8 * (long long)np)[p];
            __syncwarp();
        }
        if (lane == 0) {
            const double r = P.r[p], rho_s = P.rho_s[p];
            const double area = 3.14159265358979323846 * r * r, m = rho_s * area, wgt = (rho_s - A.bp.rho_f) * area;
            P.im[p] = 1.0 / m;
            P.iI[p] = 1.0 / (0.5 * m * r * r);
            // (1 - rho_f / rho_s) m g is (rho_s - rho_f) pi r^2 g
            P.wx[p] = wgt * A.bp.gx;
            P.wy[p] = wgt * A.bp.gy;
            P.reach[p] = r + A.ph.cut_d;
            P.rf[p] = (float)r;
        }
        __syncwarp();
        particle_advance(A, p, load_particle(A, p, cur, lane), cur, bins_at(A.B, cur, rot), false, 0,
                         A.clock ? __ldcg(&A.clock->tag) : 0u, 0.0, 0.0, lane);
    }
    if (A.clock) {
        __syncthreads();
        if (threadIdx.x == 0 && atomicAdd(left, 1u) == gridDim.x - 1) {
            *left = 0;
            A.clock->rot = rot;
        }
    }
}

// The particle update as a launch of its own (a strip's step, the static
// step), one warp per particle: phase 0: the whole update after a
// sweep_kernel; 1: only the sums of a strip's bins, to fpart; 2: the rest from
// the sums in fpart.
static __global__ void __launch_bounds__(PART_WARPS * 32)
particles_kernel(const __grid_constant__ PartArgs A, int cur, int phase) {
    const int lane = threadIdx.x & 31, p = blockIdx.x * PART_WARPS + (threadIdx.x >> 5);
    if (p >= A.bp.np) return;
    const int nxt = cur ^ 1;
    const Bins in = bins_at(A.B, cur, cur), out = bins_at(A.B, nxt, nxt);
    const int comp = component(lane);
    double f = 0.0;
    Repulsion c{0.0, 0.0};
    if (phase != 2) {
        c = pair_repulsion(A, p, cur, in, lane);
        f = hydro_sums<false>(A, p, in, 0u, lane, nullptr);
    }
    double *o = A.fpart ? A.fpart + 5 * (long long)p : nullptr;
    if (phase == 1) {
        if ((lane & 7) == 0 && comp < 3) o[comp] = f;
        if (lane == 0) { o[3] = c.x; o[4] = c.y; }
        return;
    }
    if (phase == 2) { f = o[comp < 3 ? comp : 0]; c.x = o[3]; c.y = o[4]; }
    wall_repulsion(A, p, cur, c);
    if (lane == 0) { A.fcol[2 * (long long)p] = c.x; A.fcol[2 * (long long)p + 1] = c.y; }
    particle_advance(A, p, load_particle(A, p, cur, lane), nxt, out, true, 0, 0u, f,
                     comp == 0 ? c.x : (comp == 1 ? c.y : 0.0), lane);
}

// ------------------------------------------------------------ fused steps
// One launch advances a lattice, or every lattice of a batch, by nsteps whole
// steps.  Most blocks sweep; the first few update the particles: each of their
// warps owns some, finds their repulsion at the start of a step, then watches
// their counters and updates each particle as soon as its last partial is
// counted, while the other blocks sweep on.  (Two other splits were measured
// on the 4096^2 suspension.  The warp that counts a particle's last partial
// updates it: a warp held up by one update is then the last to count on its
// next segment too, one SM ended up with a seventh of all updates, 630 us a
// step.  Each sweeping warp owns some: the update's registers and calls sit in
// the sweep's loop, 234 us.)  Between steps the blocks meet at a barrier in
// device memory (the launch is then cooperative: all blocks are resident).
//
// Row segments are dealt by tickets: a warp's first segment is fixed, each
// further one comes from a counter, taken one segment ahead.  (Dealt
// round-robin, the warps of the 4096^2 suspension finished their segments
// between 160 and 220 us into the step.)  The blocks form TICKET_GROUPS
// groups with a counter each, so that no counter is asked more than once in
// some ten nanoseconds; a group's segments lie interleaved with the others',
// which keeps all warps near the same rows.
constexpr int TICKET_GROUPS = 8;

struct GridSync {               // all 0 between launches, but for the clock and mean_tag
    unsigned arrived[2][32];    // sweeping blocks, particle blocks (a cache line each)
    unsigned left, pad0;        // blocks that have left; from bit 16 on, abandon()s
    StepClock clock;            // a context's own (a batch's launches advance its members' clocks)
    unsigned mean_tag;          // the clock's step number when the force sums were last zeroed
    unsigned pad[27];
    unsigned ticket[3][TICKET_GROUPS][32];      // by step in rotation and group, a cache line each
};

struct StepRun {
    int nsteps;
    int dry;                    // sweep only: no contribution is counted, no particle updated (autotuning)
    GridSync *sync;
    int pblocks;                // blocks that update particles
    int ahead;                  // of them, those first in the grid: all or none (see launch_steps)
};

// Thread 0 of a block: count it as arrived, and wait until `target` blocks
// have; false when the bounded wait gave up.
__device__ __forceinline__ void arrive_block(unsigned *arrived) {
    asm volatile("red.add.release.gpu.global.u32 [%0], 1;" ::"l"(arrived) : "memory");
}
__device__ __forceinline__ bool await_blocks(const unsigned *arrived, unsigned target) {
    unsigned long long t0 = 0;
    for (;;) {
        unsigned v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(arrived) : "memory");
        if ((int)(v - target) >= 0) return true;
        const unsigned long long t = global_ns();
        if (t0 == 0) t0 = t;
        else if (t - t0 > WAIT_LIMIT_NS) return false;
    }
}

// A wait ran out (or had before the launch): not all steps were done, and the
// last block out tells every lattice.  Before this block is counted out, in the
// same word: a word of its own is a trip to the L2 more at the end of each
// launch, 0.7 us of a PS step.
constexpr unsigned ABANDONED = 1u << 16;
__device__ __forceinline__ void abandon(GridSync *sync) { atomicAdd(&sync->left, ABANDONED); }

// The frame's move by s columns, in place: warps take rows of planes, 32
// columns at a time in the direction of the move (each value is read before
// its column is overwritten).
template <typename T>
__device__ __noinline__ void shift_rows(T *buf, const Lattice &L, int s, int gw, int nw, int lane) {
    for (int r = gw; r < 9 * L.ny; r += nw) {
        T *line = buf + (long long)(r / L.ny) * L.plane + (long long)(r % L.ny) * L.row;
        // the column entering: the far end on a periodic axis, else its neighbour
        const T enter = __ldcg(line + (s > 0 ? (L.per_x ? 0 : L.nx - 1) : (L.per_x ? L.nx - 1 : 0)));
        for (int b = 0; b < L.nx; b += 32) {
            const int x = s > 0 ? b + lane : L.nx - 1 - b - lane;
            const bool in = x >= 0 && x < L.nx, edge = x + s < 0 || x + s >= L.nx;
            const T v = in && !edge ? __ldcg(line + x + s) : enter;
            __syncwarp();
            if (in) line[x] = v;
            __syncwarp();
        }
    }
}

// Position in a work list: lattice, row and segment.
struct Cursor {
    int lat, y, tx;
};

// One lattice's work list.
template <typename T>
struct OneWork {
    const SweepArgs<T> &one;
    const PartArgs &pa;
    __device__ __forceinline__ const PartArgs &part(int) const { return pa; }
    __device__ __forceinline__ int items() const { return one.L.ny * one.L.ntx; }
    __device__ __forceinline__ int tiles() const { return one.L.ntx * one.L.nty; }
    __device__ __forceinline__ int parts() const { return one.np; }
    __device__ __forceinline__ const SweepArgs<T> &args(int) const { return one; }
    __device__ __forceinline__ void seek(Cursor &c, int item) const {
        c.y = row_of(item, one.ntx_inv, one.L.ntx);
        c.tx = item - c.y * one.L.ntx;
    }
    __device__ __forceinline__ int find_tile(int t, int &lat) const { lat = 0; return t; }
    __device__ __forceinline__ int find_part(int g, int &lat) const { lat = 0; return g; }
    // which populations and positions step st of the launch reads
    __device__ __forceinline__ int parity(int, int st) const { return one.cur ^ (st & 1); }
    __device__ __forceinline__ bool reversed(int st) const { return one.turn && parity(0, st); }
    __device__ __forceinline__ int lattices() const { return 1; }
};

// A batch's: the members' segments, tiles and particles, one after another.
// A warp's items only grow within a step, so its lattice is found by stepping
// on from the last one (a few lattices at most).
template <typename T>
struct BatchWork {
    const BatchArgs<T> &ba;
    __device__ __forceinline__ const PartArgs &part(int lat) const { return *ba.a[lat].pa; }
    __device__ __forceinline__ int items() const { return ba.item_start[ba.n]; }
    __device__ __forceinline__ int tiles() const { return ba.tile_start[ba.n]; }
    __device__ __forceinline__ int parts() const { return ba.part_start[ba.n]; }
    __device__ __forceinline__ const SweepArgs<T> &args(int lat) const { return ba.a[lat]; }
    __device__ __forceinline__ void seek(Cursor &c, int item) const {
        while (c.lat + 1 < ba.n && ba.item_start[c.lat + 1] <= item) ++c.lat;
        const int local = item - ba.item_start[c.lat], ntx = ba.a[c.lat].L.ntx;
        c.y = row_of(local, ba.a[c.lat].ntx_inv, ntx);
        c.tx = local - c.y * ntx;
    }
    __device__ __forceinline__ int find_tile(int t, int &lat) const {
        lat = batch_find(ba.tile_start, ba.n, t);
        return t - ba.tile_start[lat];
    }
    __device__ __forceinline__ int find_part(int g, int &lat) const {
        lat = batch_find(ba.part_start, ba.n, g);
        return g - ba.part_start[lat];
    }
    __device__ __forceinline__ int parity(int lat, int st) const { return ba.a[lat].cur ^ (st & 1); }
    __device__ __forceinline__ bool reversed(int) const { return false; }
    __device__ __forceinline__ int lattices() const { return ba.n; }
};

// May every particle have a warp of its own?  Then nothing is counted: the
// warp reads its particle's partials until they carry the step's tag, and has
// all else that the update needs at hand before.  (A count costs the chain of
// a small lattice's step two more trips to the L2.)
template <typename WORK>
__device__ __forceinline__ bool own_warps(const WORK &wk, int npw) { return wk.parts() <= npw; }

// The particle blocks' part of a step: warp pw of npw.
template <typename WORK>
__device__ __forceinline__ bool update_particles(const WORK &wk, const StepClock *clk, int st, int shift, int pw, int npw,
                                                 int lane) {
    const int total = wk.parts();
    const bool own = own_warps(wk, npw);
    bool late = false;
    Repulsion c{0.0, 0.0};
    for (int g = pw; g < total; g += npw) {
        int lat;
        const int p = wk.find_part(g, lat);
        const PartArgs &A = wk.part(lat);
        c = pair_repulsion(A, p, wk.parity(lat, st), bins_at(A.B, wk.parity(lat, st), (clk[lat].rot + st) % 3), lane);
        wall_repulsion(A, p, wk.parity(lat, st), c);
        if (lane == 0) {
            A.fcol[2 * (long long)p] = c.x;
            A.fcol[2 * (long long)p + 1] = c.y;
        }
    }
    __syncwarp();        // (the same warp reads them below)
    // up to 32 of the warp's particles at a time, one watched by each lane
    for (int g0 = pw; g0 < total; g0 += 32 * npw) {
        const int g = g0 + lane * npw;
        int lat = 0, p = -1;
        const int *done = nullptr;
        if (g < total) {
            p = wk.find_part(g, lat);
            const PartArgs &A = wk.part(lat);
            done = A.B.done + (long long)wk.parity(lat, st) * A.B.parts + p;
        }
        unsigned long long t0 = global_ns();
        while (__any_sync(0xffffffffu, done != nullptr)) {
            unsigned ready = __ballot_sync(0xffffffffu, done != nullptr && (own || load_done(done) == 0));
            if (ready == 0) {
                if (__any_sync(0xffffffffu, global_ns() - t0 > WAIT_LIMIT_NS)) return false;
                __nanosleep(100);
                continue;
            }
            if (ready >> lane & 1u) done = nullptr;
            for (; ready; ready &= ready - 1) {
                const int l = __ffs(ready) - 1;
                const int q = __shfl_sync(0xffffffffu, p, l), ql = __shfl_sync(0xffffffffu, lat, l);
                const PartArgs &A = wk.part(ql);
                const int cur = wk.parity(ql, st), rot = (clk[ql].rot + st) % 3;
                const unsigned tag = clk[ql].tag + st;
                const PartState ps = load_particle(A, q, cur, lane);
                const int comp = component(lane);
                double ca = comp == 0 ? c.x : (comp == 1 ? c.y : 0.0);
                if (!own && comp < 2) ca = __ldcg(A.fcol + 2 * (long long)q + comp);
                const double f = hydro_sums<true>(A, q, bins_at(A.B, cur, rot), tag, lane, &late);
                if (late) return false;
                particle_advance(A, q, ps, cur ^ 1, bins_at(A.B, cur ^ 1, rot3(rot + 1)), true, shift, tag + 1, f, ca, lane);
            }
            t0 = global_ns();
        }
    }
    return true;
}

// HALVES: two warps share each row segment, one pass each, where that still
// leaves every warp at most one: a step of such a lattice is as long as a
// warp's chain through its segment.  (us per step: 200 x 100 cylinder 9.3 ->
// 8.3, 501 x 101 channel with a moving frame 10.9 -> 9.9.  A kernel of its own:
// decided at run time, it took 15 % from every other lattice.)
template <typename T, bool EDGES, int W, bool PS, int LATTICES, bool HALVES, typename WORK>
__device__ __forceinline__ void run_steps(const WORK &wk, const PartArgs *frame, const StepRun &run) {
    extern __shared__ __align__(128) unsigned char smem_raw[];
    __shared__ StepClock clk[LATTICES]; // every lattice's clock as the launch starts
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    SweepSmem<T, W> sm(smem_raw, warp);
    Ring ring{sm.bar, 0u, false};
    if (lane == 0) {
        mbar_init(ring.bar, 1);
        mbar_fence_init();
    }
    // A lattice whose steps were given up once takes no more of them: what its
    // particles would wait for is not there.
    bool dead = false;
    for (int k = threadIdx.x; k < wk.lattices(); k += blockDim.x) {
        clk[k].tag = __ldcg(&wk.args(k).clock->tag);
        clk[k].rot = __ldcg(&wk.args(k).clock->rot);
        dead |= __ldcg(wk.args(k).err) & ERR_TIMEOUT;
    }
    int st = __syncthreads_or(dead) ? run.nsteps + 1 : 0;
    // this block among the sweeping ones (from nsb on: a particle block), its group
    // and the group's warps
    const int nsb = (int)gridDim.x - run.pblocks;
    const int sb = (int)blockIdx.x >= run.ahead ? (int)blockIdx.x - run.ahead : nsb + (int)blockIdx.x;
    const bool sweeps = sb < nsb;
    const int ngroups = nsb < TICKET_GROUPS ? nsb : TICKET_GROUPS;
    const int group = sb % ngroups, gwarps = (nsb / ngroups + (group < nsb % ngroups)) * W;
    auto item_of = [&](int k) { return ((k / W) * ngroups + group) * W + (k & (W - 1)); };
    const int nitems = wk.items() << (int)HALVES;
    const bool counted = !run.dry && !own_warps(wk, run.pblocks * W);
    const FieldsOut fo{nullptr, nullptr, nullptr, nullptr};
    unsigned target[2] = {0, 0};        // arrivals that end the present meeting
    // Between steps the blocks meet: what they have written is then visible,
    // also to the bulk copies (the async proxy).  A warp that gave up (`bad`)
    // takes its block out; the others' bounded waits then end, and the launch:
    // every lattice in it misses steps, and its error word says so.
    auto arrive = [&](bool bad) {
        if (sweeps) asm volatile("fence.proxy.async;" ::: "memory");
        if (__syncthreads_or(bad)) return false;
        target[0] += (unsigned)nsb;
        target[1] += (unsigned)run.pblocks;
        if (threadIdx.x == 0) arrive_block(run.sync->arrived[sweeps ? 0 : 1]);
        return true;
    };
    auto await = [&](int which) {
        bool bad = false;
        if (threadIdx.x == 0) bad = !await_blocks(run.sync->arrived[which], target[which]);
        if (__syncthreads_or(bad)) return false;
        asm volatile("fence.proxy.async;" ::: "memory");
        return true;
    };
    // the warp's first segment of a step, its copy issued
    Cursor c{0, 0, 0};
    T wv = T();             // the staged segment's periodic-edge value (wrap_load)
    int item = 0;
    bool have = false;
    auto open_step = [&](int st) {
        c = Cursor{0, 0, 0};
        item = item_of((sb / ngroups) * W + warp);
        have = item < nitems;
        if (!have) return;
        if (wk.reversed(st)) item = nitems - 1 - item;
        wk.seek(c, item >> (int)HALVES);
        const SweepArgs<T> &a = wk.args(c.lat);
        const T *src = a.buf[wk.parity(c.lat, st)];
        const int ys = streamed_row<EDGES>(a.L, c.y);
        issue_segment<T>(src, a.L, ys, c.tx, sm.stage, ring.bar, lane);
        wv = wrap_load<T>(src, a.L, ys, c.tx, lane);
        ring.pending = true;
    };

    if (sweeps && st == 0) open_step(0);
    for (; st < run.nsteps; ++st) {
        bool timed_out = false;
        int shift = 0;
        const int track = frame ? frame->track : -1;    // (a batch's frames stand still)
        if (track >= 0) {
            const PartArgs &f = *frame;
            shift = frame_move(__ldcg((wk.parity(0, st) ? f.P.x[1] : f.P.x[0]) + f.track), f.track_x, f.L.nx, f.L.per_x);
        }
        if (!sweeps) {
            if (!run.dry && !update_particles(wk, clk, st, shift, (sb - nsb) * W + warp, run.pblocks * W, lane)) {
                if (lane == 0) abandon(run.sync);
                timed_out = true;
            }
        } else {
            unsigned *ticket = &run.sync->ticket[st % 3][group][0];
            if (warp == 0 && lane == 0 && sb < ngroups) run.sync->ticket[(st + 2) % 3][group][0] = 0;
            if (!run.dry && wk.parts() > 0) {
                // the counts the step after next adds to
                for (int t = sb * blockDim.x + threadIdx.x; t < wk.tiles(); t += nsb * blockDim.x) {
                    int lat;
                    const int tl = wk.find_tile(t, lat);
                    const SweepArgs<T> &a = wk.args(lat);
                    if (a.np > 0) a.B.count[(long long)((clk[lat].rot + st + 2) % 3) * a.B.tiles + tl] = 0;
                }
            }
            while (have) {
                int k = 0;
                if (lane == 0) k = gwarps + (int)atomicAdd(ticket, 1u);
                item = item_of(__shfl_sync(0xffffffffu, k, 0));
                have = item < nitems;
                if (wk.reversed(st)) item = nitems - 1 - item;
                Cursor nx = c;
                if (have) wk.seek(nx, item);
                const SweepArgs<T> &a = wk.args(c.lat), &an = wk.args(nx.lat);
                const int cur = wk.parity(c.lat, st);
                if (!sweep_segment<T, MODE_STEP, EDGES, PS, true, HALVES>(
                        a, a.buf[cur], a.buf[cur ^ 1], bins_at(a.B, cur, (clk[c.lat].rot + st) % 3), c.y, c.tx, sm.stage,
                        ring, have, an.buf[wk.parity(nx.lat, st)], an.L, nx.y, nx.tx, sm.crec, sm.cid, wv,
                        clk[c.lat].tag + st - run.dry, counted, fo, lane,
                        warp & 1)) {
                    if (lane == 0) abandon(run.sync);
                    timed_out = true;
                    break;
                }
                c = nx;
            }
        }
        if (run.nsteps == 1) {      // (`continue`, the same, took the FP16 step 202.0 us on 4096^2; this, 198.3)
            st = 1;
            break;
        }
        const bool more = st + 1 < run.nsteps;
        if (shift != 0) {
            if (!arrive(timed_out) || !await(0) || !await(1)) break;
            shift_rows<T>(wk.args(0).buf[wk.parity(0, st) ^ 1], wk.args(0).L, shift, (int)blockIdx.x * W + warp,
                          (int)gridDim.x * W, lane);
            if (blockIdx.x == 0 && threadIdx.x == 0) *frame->frame_off = __ldcg(frame->frame_off) + shift;
            asm volatile("fence.proxy.async;" ::: "memory");        // (the particle blocks moved rows too)
        }
        if (more) {
            // the populations are there once the sweeping blocks have met, and
            // the next step's first copies start; the bins and positions follow
            if (!arrive(timed_out) || !await(0)) break;
            if (shift != 0 && !await(1)) break;         // (every block moved rows)
            if (sweeps) open_step(st + 1);
            if (shift == 0 && !await(1)) break;
        }
    }
    // let the copies this warp still has in flight (it gave up, or its block
    // left) land before the block releases its shared memory (the wait bounded)
    if (ring.pending) mbar_wait_bounded(ring.bar, ring.parity);
    // the last block out leaves the counters as it found them, and advances the clocks
    __syncthreads();
    if (threadIdx.x == 0 && st != run.nsteps) abandon(run.sync);        // (left before its end)
    const unsigned left = threadIdx.x == 0 ? atomicAdd(&run.sync->left, 1u) : 0u;
    if (threadIdx.x == 0 && left % ABANDONED == gridDim.x - 1) {
        run.sync->arrived[0][0] = run.sync->arrived[1][0] = 0;
        run.sync->left = 0;
        if (left >= ABANDONED)
            for (int k = 0; k < wk.lattices(); ++k) atomicOr(wk.args(k).err, ERR_TIMEOUT);
        for (int q = 0; q < 3; ++q)
            for (int g = 0; g < TICKET_GROUPS; ++g) run.sync->ticket[q][g][0] = 0;
        for (int k = 0; k < wk.lattices() && !run.dry; ++k) {
            StepClock *c = wk.args(k).clock;
            c->tag = clk[k].tag + (unsigned)run.nsteps;
            c->rot = (clk[k].rot + run.nsteps) % 3;
        }
    }
}

template <typename T, bool EDGES, int W, bool PS = false, bool HALVES = false>
__global__ void __launch_bounds__(W * 32, sm_warps<T>() / W)
step_kernel(const __grid_constant__ SweepArgs<T> one, const __grid_constant__ PartArgs pa,
            const __grid_constant__ StepRun run) {
    const OneWork<T> wk{one, pa};
    run_steps<T, EDGES, W, PS, 1, HALVES>(wk, &pa, run);
}

template <typename T, int W>
__global__ void __launch_bounds__(W * 32, sm_warps<T>() / W)
step_batch_kernel(const __grid_constant__ BatchArgs<T> ba, const __grid_constant__ StepRun run) {
    const BatchWork<T> wk{ba};
    run_steps<T, true, W, false, BATCH_LAUNCH_MAX, false>(wk, nullptr, run);
}

// ------------------------------------------------------------ conversions
// e_i of direction i given at run time (the conversion kernels index by a
// computed direction).
__device__ __forceinline__ float ref_e_of(const Lattice &L, int i) {
    float v = L.ref_e[0];
#pragma unroll
    for (int j = 1; j < 9; ++j)
        if (i == j) v = L.ref_e[j];
    return v;
}

// Populations <-> FP64 f_i (dense 9 x ny x nx) for checkpoints.
template <typename T>
__global__ void export_kernel(const T *__restrict__ src, Lattice L, double *__restrict__ out) {
    const long long n = (long long)L.nx * L.ny;
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < 9 * n; k += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(k / n);
        const long long r = k - i * n;
        const int y = (int)(r / L.nx), x = (int)(r - (long long)y * L.nx);
        const double v = (double)Storage<T>::load1(src + i * L.plane + (long long)y * L.row + x);
        out[k] = (std::is_same<T, float>::value ? v : v * (double)L.ref_q + (double)ref_e_of(L, i)) + (double)wof(i);
    }
}

template <typename T>
__global__ void import_kernel(T *__restrict__ dst, Lattice L, const double *__restrict__ in) {
    const long long n = (long long)L.nx * L.ny;
    // the same FP32 weights the deviations are taken against, so that an
    // exported state imports back bit for bit
    const double w[9] = {wof(0), wof(1), wof(2), wof(3), wof(4), wof(5), wof(6), wof(7), wof(8)};
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < 9 * n; k += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(k / n);
        const long long r = k - i * n;
        const int y = (int)(r / L.nx), x = (int)(r - (long long)y * L.nx);
        const double dv = in[k] - w[i];
        Storage<T>::store1(dst + i * L.plane + (long long)y * L.row + x,
                           std::is_same<T, float>::value ? (float)dv
                                                         : (float)((dv - (double)ref_e_of(L, i)) * (double)L.ref_iq));
    }
}

// Uniform initial state f^eq(rho0, u0) written as deviations on every node.
// PS-LBM (Sec. 2.2): the covered area of every cell about each particle
// (B = eps_s, Eq. 8), once per step after the particle update, for the next
// sweep to look up.  Particle p's table holds the (2K+1)^2 cells about
// (floor X, floor Y), row-major; the cell at offset (i, j) is the node
// (floor X + i, floor Y + j).  The same decisions as the sweep's: 0 beyond
// the reach r + cut, 1 once every corner is inside.  One block per particle
// walks its table; the particle's fractional centre is formed once in FP64
// and shared as FP32 hi + lo.  The cells the circle crosses (about one in
// eight, scattered over every warp) are gathered first and then summed by
// whole warps; cells past the list's capacity (only for very large discs)
// are summed where they are found.
constexpr int COVER_BX = 32, COVER_BY = 8, COVER_RING = 2048;

static __global__ void __launch_bounds__(COVER_BX * COVER_BY)
cover_kernel(float *__restrict__ cover, const double *__restrict__ xs, const double *__restrict__ ys,
             const double *__restrict__ rs, int np, Physics ph) {
    __shared__ int ring[COVER_RING];
    __shared__ int nring;
    __shared__ float frac[5];               // x - floor x (hi, lo), y - floor y (hi, lo), r
    const int tid = threadIdx.y * COVER_BX + threadIdx.x;
    const int K = ph.ck, S = 2 * K + 1;
    for (int p = blockIdx.x; p < np; p += gridDim.x) {
        if (tid == 0) {
            nring = 0;
            const double X = xs[p], Y = ys[p];
            const double fx = X - floor(X), fy = Y - floor(Y);
            frac[0] = (float)fx;
            frac[1] = (float)(fx - (double)frac[0]);
            frac[2] = (float)fy;
            frac[3] = (float)(fy - (double)frac[2]);
            frac[4] = (float)rs[p];
        }
        __syncthreads();
        const float rf = frac[4], Rf = rf + ph.cut;
        float *tab = cover + (long long)p * S * S;
        for (int iy = threadIdx.y; iy < S; iy += COVER_BY) {
            const float dy = ((float)(iy - K) - frac[2]) - frac[3];
            for (int ix = threadIdx.x; ix < S; ix += COVER_BX) {
                const float dx = ((float)(ix - K) - frac[0]) - frac[1];
                const float d2 = dx * dx + dy * dy;
                float v = 0.f;
                bool crossed = false;
                if (d2 <= Rf * Rf) {
                    const float l = rf - sqrtf(d2);
                    if (l >= ph.cut) v = 1.0f;
                    else crossed = l >= -ph.cut;
                }
                if (crossed) {
                    const int slot = atomicAdd(&nring, 1);
                    if (slot < COVER_RING) ring[slot] = iy * S + ix;
                    else tab[iy * S + ix] = cell_cover(dx, dy, rf);
                } else {
                    tab[iy * S + ix] = v;
                }
            }
        }
        __syncthreads();
        const int nr = nring < COVER_RING ? nring : COVER_RING;
        for (int k = tid; k < nr; k += COVER_BX * COVER_BY) {
            const int j = ring[k], cy = j / S, cx = j - cy * S;
            const float dx = ((float)(cx - K) - frac[0]) - frac[1], dy = ((float)(cy - K) - frac[2]) - frac[3];
            tab[j] = cell_cover(dx, dy, rf);
        }
        __syncthreads();
    }
}

// Moving computational domain (Sec. 3.5): when the frame moves by s columns
// (decided from the tracked particle's x at the start of the step that just
// ran, as the particle update decided it), column x of every population
// plane takes the stored values of column x + s: rolled on a periodic x
// axis, otherwise clamped, so the entering column repeats its neighbour.
// The move is in place, one row of one plane at a time through shared
// memory (nx elements); block 0 adds s to the frame offset.
template <typename T>
__global__ void frame_shift_kernel(T *__restrict__ buf, Lattice L, const double *__restrict__ xt, int track,
                                   double track_x, long long *__restrict__ offset) {
    extern __shared__ __align__(16) unsigned char frame_row[];
    T *row = reinterpret_cast<T *>(frame_row);
    const int s = frame_move(xt[track], track_x, L.nx, L.per_x);
    if (s == 0) return;
    if (blockIdx.x == 0 && threadIdx.x == 0) *offset += s;
    for (int y = blockIdx.x; y < L.ny; y += gridDim.x) {
        for (int i = 0; i < 9; ++i) {
            T *line = buf + (long long)i * L.plane + (long long)y * L.row;
            for (int x = threadIdx.x; x < L.nx; x += blockDim.x) row[x] = line[x];
            __syncthreads();
            for (int x = threadIdx.x; x < L.nx; x += blockDim.x) {
                int src = x + s;
                if (L.per_x) src = src < 0 ? src + L.nx : (src >= L.nx ? src - L.nx : src);
                else src = src < 0 ? 0 : (src > L.nx - 1 ? L.nx - 1 : src);
                line[x] = row[src];
            }
            __syncthreads();
        }
    }
}

template <typename T>
__global__ void init_kernel(T *__restrict__ dst, Lattice L, float drho, float ux, float uy) {
    const long long n = (long long)L.nx * L.ny;
    float e[9];
    eq_dev9(drho, 1.0f + drho, ux, uy, e);
    for (long long k = blockIdx.x * (long long)blockDim.x + threadIdx.x; k < 9 * n; k += (long long)gridDim.x * blockDim.x) {
        const int i = (int)(k / n);
        const long long r = k - i * n;
        const int y = (int)(r / L.nx), x = (int)(r - (long long)y * L.nx);
        float v = e[0];
#pragma unroll
        for (int j = 1; j < 9; ++j)
            if (i == j) v = e[j];
        // (16-bit storage: the initial state is the reference state itself, s_i = 0)
        Storage<T>::store1(dst + i * L.plane + (long long)y * L.row + x, std::is_same<T, float>::value ? v : 0.0f);
    }
}

}  // namespace dilbm
