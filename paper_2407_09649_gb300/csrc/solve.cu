// solve.cu -- batched GP instances: K assembly, FP64 Cholesky, alpha, and the fused
// evaluation of every query of the instance (latent mean Eq. 1, variance Eq. 2, gradient
// Eq. 5, reverting Eq. 3 and distance variance Eq. 4), plus the backward pass.
//
// A CTA (or a cluster of them, see group_ctas) works on one instance at a time and takes instances
// from a list sorted by decreasing size (a persistent launch per size bucket, longest first).
// Plain kernel: A = K + sigma^2 I is stored as the lower triangle of 8x8 tiles (64 contiguous
// doubles per tile, tiles in packed row order), in shared memory when it fits, else in a per-CTA
// global workspace; the Cholesky factorisation is right-looking by 8-column panels, all on the
// FP64 pipe.  FP64 mma.sync (m8n8k4) is not used: it runs at the same FP64 rate and its results are
// those of the ascending fma chain, but one holds a sub-partition's pipe for 580 clocks, against
// 66 for an FMA, so every chain beside it waits.  Emulated kernel: see factor_emulated.
#include <algorithm>
#include <cstdio>
#include <cstring>
#include <vector>

#include "internal.h"

namespace vgp {

namespace {

// offset of tile (it, jt), jt <= it, in the tile-packed lower triangle
__host__ __device__ __forceinline__ int64_t tix(int it, int jt) { return ((int64_t)it * (it + 1) / 2 + jt) * 64; }
__host__ __device__ __forceinline__ int64_t n_tiles(int nt) { return (int64_t)nt * (nt + 1) / 2; }

// The emulated kernel's matrix: lower triangle of 32x32 blocks of 1024 words, in packed row order.
// A block holds either the fixed point (kFixBits), column by column (word 32 c + r), so that the
// trailing update's warps, one row per lane, read and write whole 256-byte lines; or, once its
// columns are reached, 8x8 FP64 tiles, tile column by tile column.  In both forms 16 columns
// take the same half of the block, so the warp that owns a half turns it from one into the other.
__host__ __device__ __forceinline__ int64_t bix(int bi, int bj) { return ((int64_t)bi * (bi + 1) / 2 + bj) * 1024; }
__host__ __device__ __forceinline__ int64_t n_blocks(int rows) {
    const int64_t nb = (rows + 31) / 32;
    return nb * (nb + 1) / 2;
}
// offset of the FP64 tile (it, jt), jt <= it, of the emulated kernel's matrix
__host__ __device__ __forceinline__ int64_t eix(int it, int jt) {
    return bix(it >> 2, jt >> 2) + ((jt & 3) * 4 + (it & 3)) * 64;
}
constexpr int kTileCol = 256;  // words from a tile to its right neighbour in the block

// Position of element (r, c) inside a 64-double tile: row major with the columns of rows
// 2, 3, 6, 7 XOR-swizzled by 4, so the loads of a warp's 32 lanes at (row lane / 4, column
// lane % 4) hit distinct shared-memory banks in each half-warp.
__host__ __device__ __forceinline__ int te(int r, int c) { return r * 8 + (c ^ ((r & 2) << 1)); }

// row index of packed-triangle entry p (0 <= col <= row)
__device__ __forceinline__ int tri_row(int p) {
    int r = (int)((sqrtf(8.0f * (float)p + 1.0f) - 1.0f) * 0.5f);
    while ((r + 1) * (r + 2) / 2 <= p) ++r;
    while (r * (r + 1) / 2 > p) --r;
    return r;
}

constexpr int kEmuThreads = 256;  // CTA size of the emulated-update kernels (two CTAs per SM)
// Largest CTA of the plain kernels: five warps per sub-partition leave each thread 96 registers (k_solve is
// bounded to them; k_backward takes 86, and 96 with spills when bounded).  A chosen shape of more
// threads runs with this many.
constexpr int kPlainThreads = 640;
constexpr int kEB = 4;            // tiles (of 8 columns) per block of the emulated factorisation
constexpr int kEK = kEB / 2;      // 16-column mma steps per block
constexpr int kDiagTiles = kEB * (kEB + 1) / 2;

struct SolveCtx {
    SolveBatch b;
    DevParams P;
    int* err;
    int* counter;
    const int32_t* order;  // instance ids, decreasing N (null: inst_base + work index)
    int inst_base;
    int n_work;
    const int* plan;       // device bucket plan (graph mode): counts [5], then offsets [5]
    int bucket;
    int npad;              // largest N in this launch, rounded up to 8
    int a_in_smem;
    int stage_panel;       // A global: current panel column staged in shared memory
    double* ws_a;          // per-CTA tile-packed A when not in shared memory
    int64_t ws_a_stride;
    double* ws_v;          // per-CTA variance columns [npad][blockDim]
    int64_t ws_v_stride;
    uint8_t* ws_e;         // per-CTA bf16 slices and row scales (emulated trailing updates)
    int64_t ws_e_stride;
    BackwardBatch bw;
    const int* chunk_off = nullptr;  // work items (see k_chunk_plan): chunk offsets over the order;
                                     // nullptr: one work item per instance
    const int* chunk_q = nullptr;    // queries of a work item for this launch (0: all of them; chunk_len)
    int chunk_qn = 0, chunk_cap = 0;
    int qmax = 0;          // emulated kernel with variance: query rows appended to A (0: none)
    int nrow = 0;          // emulated kernel: rows of the workspace matrices (npad + qmax)
    int ncta = 1;          // emulated kernel: CTAs (a cluster) that work on one instance together
};

struct Shared {
    double* X;      // [N][3] local FP64
    double* alpha;  // [npad]
    double* invd;   // [npad] 1 / L_ii
    double* z;      // [npad] scratch
    double* w;      // [npad] scratch (backward pass only)
    double* Tinv;   // [64] inverse of the current diagonal tile
    double* T256;   // [256] 2^(j/256) for exp_neg
    double* A;      // tile-packed lower triangle
    double* panel;  // [npad/8 - 1][64] current panel column when A is in global memory
    float* Xf;      // [N][3]
    float* alf;     // [npad] alpha rounded to FP32
    float* alf_lo;  // [npad] alpha - alf, rounded to FP32
    int* xi;        // [npad] lattice offsets x | y << 8 | z << 16 (lattice instances)
    double* pa[4];  // property weights per channel (property mode): channels 0 and 1 reuse the
                    // distance alpha and its FP32 copies, which that mode does not use
    double* Tblk;   // [kEB][64] inverses of the diagonal tiles of the current block
    uint8_t* dtab;  // [8][32] entries of the diagonal tiles' updates (diag_entry)
    double* Dsc;    // [64] plain kernel, A in global memory: the current diagonal tile
    double* Dblk;   // [kDiagTiles][64] the current block's diagonal tiles (packed lower triangle)
    unsigned char* stage;  // emulated kernel: slice operands of the tensor-core updates (aliases
                           // X .. alf_lo, which the factorisation does not use; reloaded after it)
    float* qw;             // emulated kernel: [kBorderQ][3] world coordinates of appended queries (FP32;
                           // NaN: not finite); lattice instances: [0] the lattice code's bits, [1] NaN
                           // when not finite
    double* Dsol;          // emulated kernel: [2][kDiagTiles][64] a group's diagonal tiles in the solves
    float* Xw;             // emulated kernel: [npad][3] world coordinates of the points (FP32, exact)
    float2* Tff;           // emulated kernel: 2^(j/256), j = 0..255, as float pairs
};

// Emulated trailing updates on the tensor cores (tcgen05): an output tile is kBandT row tiles
// (128 rows, the MMA's M) by kColT row tiles (32 columns, its N) of the trailing matrix; the
// slices of one 16-column half of the block are staged for the band (A) and the column tile (B).
constexpr int kBandT = 16;
constexpr int kColT = 4;
constexpr int kSliceBytes = 2 * 2 * 128;           // one slice of a row tile: 2 K halves x 2 core matrices
constexpr int kSliceTileBytes = 7 * kSliceBytes;   // the 7 slices of a row tile
// Slices in the workspace and of a column tile (B): [group of kColT row tiles][slice][row tile], so a
// column tile is one contiguous copy.  The band's slices (A) are staged [slice][row tile].
constexpr int kGroupBytes = kColT * kSliceTileBytes;
constexpr int kStageA = kBandT * kSliceTileBytes;
constexpr int kStageB = kGroupBytes;
constexpr int kStageBytes = kStageA + 2 * kStageB;
constexpr int kEmuTmemCols = 8 * 8 * kColT;    // 8 slice groups x 32 FP32 columns
// Latent variance in the emulated kernel: up to kBorderQ queries of an instance append their
// kernel vectors to A as rows, so the factorisation itself yields 1 - |L^-1 k|^2 (see
// fit_instance); an instance with more queries is factorised once per chunk of kBorderQ.
// Instances gather the queries of several query leaves (those that fall back to a shared
// leaf), so the bound is set high: a factorisation costs about N^3/6 products against
// N^2/2 per appended row.
constexpr int kBorderQ = 1024;
constexpr int kEmuCtasPerSm = 512 / kEmuTmemCols;  // CTAs whose tensor memory fits one SM

__host__ __device__ __forceinline__ size_t align128(size_t x) { return (x + 127) & ~(size_t)127; }
__host__ __device__ __forceinline__ size_t emu_fixed_bytes(int npad) {
    // invd, Tblk, Tff, Dblk, dtab
    return align128((size_t)(npad + kEB * 64 + 256 + kDiagTiles * 64 + 32) * sizeof(double));
}
__host__ __device__ __forceinline__ size_t emu_point_bytes(int npad, int nprop, bool lattice) {
    return (size_t)5 * npad * sizeof(double) + (size_t)5 * npad * sizeof(float) +
           (lattice ? (size_t)npad * sizeof(int) : 0) + (size_t)(nprop > 2 ? nprop - 2 : 0) * npad * sizeof(double);
}
// the points (also as FP32 world coordinates) and the appended queries (both forms)
__host__ __device__ __forceinline__ size_t emu_alias_bytes(int npad, int nprop, bool lattice) {
    const size_t b = emu_point_bytes(npad, nprop, lattice) + (lattice ? 0 : (size_t)3 * npad * sizeof(float)) +
                     (size_t)kBorderQ * 3 * sizeof(float);
    return b > (size_t)kStageBytes ? b : (size_t)kStageBytes;
}

// Emulated kernel: invd, the exp table and the diagonal block first, then (128-byte aligned) the
// staging buffer of the tensor-core updates, which X, alpha, z, Xf, alf, alf_lo, xi and the property
// weights alias, and so does the warps' scratch of the rows below (kEB tiles each).
__device__ Shared carve_emu(double* sm, int npad, double* ws_a, int nprop, bool lattice) {
    Shared s;
    s.invd = sm;
    s.Tblk = s.invd + npad;
    s.T256 = nullptr;  // (mixed values come from Tff, FP64 ones from exp)
    s.Tinv = nullptr;
    s.w = nullptr;
    s.panel = nullptr;
    s.A = ws_a;
    s.stage = reinterpret_cast<unsigned char*>(sm) + emu_fixed_bytes(npad);
    s.X = reinterpret_cast<double*>(s.stage);
    s.alpha = s.X + 3 * npad;
    s.z = s.alpha + npad;
    s.Xf = reinterpret_cast<float*>(s.z + npad);
    s.alf = s.Xf + 3 * npad;
    s.alf_lo = s.alf + npad;
    s.xi = lattice ? reinterpret_cast<int*>(s.alf_lo + npad) : nullptr;
    double* extra = reinterpret_cast<double*>(reinterpret_cast<int*>(s.alf_lo + npad) + (lattice ? npad : 0));
    s.pa[0] = s.alpha;
    s.pa[1] = reinterpret_cast<double*>(s.alf);
    s.pa[2] = nprop > 2 ? extra : nullptr;
    s.pa[3] = nprop > 3 ? extra + npad : nullptr;
    // world coordinates of the points off the lattice only (lattice values come from tables)
    float* after = reinterpret_cast<float*>(s.stage + emu_point_bytes(npad, nprop, lattice));
    s.Xw = lattice ? nullptr : after;
    s.qw = lattice ? after : after + 3 * npad;
    s.Tff = reinterpret_cast<float2*>(s.Tblk + kEB * 64);
    s.Dblk = s.Tblk + kEB * 64 + 256;
    s.dtab = reinterpret_cast<uint8_t*>(s.Dblk + kDiagTiles * 64);
    s.Dsc = nullptr;
    // the solves' diagonal tiles go where the world coordinates were (used by the assembly only)
    s.Dsol = reinterpret_cast<double*>(after);
    return s;
}

__device__ Shared carve(double* sm, int npad, int a_in_smem, double* ws_a, int nprop, int stage_panel,
                        bool lattice, bool with_w, bool emu = false) {
    if (emu) return carve_emu(sm, npad, ws_a, nprop, lattice);
    Shared s;
    s.stage = nullptr;
    s.qw = nullptr;
    s.Xw = nullptr;
    s.Tff = nullptr;
    s.X = sm;
    s.alpha = s.X + 3 * npad;
    s.invd = s.alpha + npad;
    s.z = s.invd + npad;
    s.w = with_w ? s.z + npad : nullptr;
    s.Tinv = s.z + (with_w ? 2 : 1) * npad;
    s.T256 = s.Tinv + 64;
    s.dtab = reinterpret_cast<uint8_t*>(s.T256 + 256);
    double* end = s.T256 + 256 + 32;
    s.Dsc = nullptr;
    s.Tblk = nullptr;
    s.Dblk = nullptr;
    s.Dsol = nullptr;
    if (a_in_smem) {
        s.A = end;
        end += n_tiles(npad / 8) * 64;
        s.panel = nullptr;
    } else {
        s.A = ws_a;
        s.Dsc = end;
        end += 64;
        s.panel = stage_panel ? end : nullptr;
        if (stage_panel) end += (int64_t)(npad / 8) * 64;
    }
    s.Xf = reinterpret_cast<float*>(end);
    s.alf = s.Xf + 3 * npad;
    s.alf_lo = s.alf + npad;
    s.xi = lattice ? reinterpret_cast<int*>(s.alf_lo + npad) : nullptr;
    double* extra = reinterpret_cast<double*>(reinterpret_cast<int*>(s.alf_lo + npad) + (lattice ? npad : 0));
    // (4 npad bytes of xi keep 8-byte alignment: npad is a multiple of 8)
    s.pa[0] = s.alpha;
    s.pa[1] = reinterpret_cast<double*>(s.alf);  // alf, alf_lo: 2 npad floats, 8-byte aligned
    s.pa[2] = nprop > 2 ? extra : nullptr;
    s.pa[3] = nprop > 3 ? extra + npad : nullptr;
    return s;
}

__host__ size_t smem_bytes(int npad, int a_in_smem, int nprop, int stage_panel, bool lattice, bool with_w = false,
                          bool emu = false) {
    if (emu) return emu_fixed_bytes(npad) + emu_alias_bytes(npad, nprop, lattice);
    size_t d = (size_t)(with_w ? 7 : 6) * npad + 64 + 256 + 32 +
               (a_in_smem ? (size_t)n_tiles(npad / 8) * 64 : 64 + (stage_panel ? (size_t)(npad / 8) * 64 : 0));
    return d * sizeof(double) + (size_t)5 * npad * sizeof(float) + (lattice ? (size_t)npad * sizeof(int) : 0) +
           (size_t)std::max(nprop - 2, 0) * npad * sizeof(double);
}

__device__ __forceinline__ int lat_m(int a, int b) {
    const int dx = (a & 255) - (b & 255), dy = ((a >> 8) & 255) - ((b >> 8) & 255), dz = ((a >> 16) & 255) - ((b >> 16) & 255);
    return dx * dx + dy * dy + dz * dz;
}

// SE kernel value of a pair of training points (Sec. III-A), FP64: from the exact lattice
// table for voxel-centre instances, else exp_neg (mixed) or the library exp (plain) of kval_arg.
__device__ __forceinline__ double kval_arg(const DevParams& P, const Shared& s, int i, int j) {
    double dx = s.X[3 * i] - s.X[3 * j], dy = s.X[3 * i + 1] - s.X[3 * j + 1], dz = s.X[3 * i + 2] - s.X[3 * j + 2];
    return -(dx * dx + dy * dy + dz * dz) * P.inv2l2;
}
__device__ __forceinline__ double kval_pair(const DevParams& P, const Shared& s, bool lattice, int i, int j) {
    if (lattice) return P.lat_tab[lat_m(s.xi[i], s.xi[j])];
    const double y = kval_arg(P, s, i, j);
    return P.precision == VGP_MIXED ? exp_neg(y, s.T256) : exp(y);
}

// ---- the emulated kernel's matrix in fixed point -------------------------------------------
// Until its column block is reached, an entry of the emulated factorisation is held as the
// integer round(v 2^61) (|v| <= 1 + sigma^2: every entry of K + sigma^2 I and of its Schur
// complements is bounded by the largest diagonal entry).  The trailing updates then subtract
// integers (one shift and one 64-bit subtraction per entry) and the block's columns are
// turned into FP64 once, by the update that completes them.  Resolution 2^-61, far below the
// updates' own rounding (2^-55 of the row maxima).
constexpr int kFixBits = 61;
__device__ __forceinline__ long long fix_of_double(double v) { return __double2ll_rn(v * 0x1p61); }
// f 2^-61 as FP64: the conversion, then the exponent lowered by 61 on the integer pipe
// (|f| >= 1 keeps the result normal)
__device__ __forceinline__ double double_of_fix(long long f) {
    return f == 0 ? 0.0 : __longlong_as_double(__double_as_longlong(__ll2double_rn(f)) - (61ll << 52));
}

// round(x 2^e) of a float x, |x| 2^e < 2^62, on the integer pipe (ties away from zero; 0 for
// subnormal x).
__device__ __forceinline__ long long fix_of_float(float x, int e) {
    const unsigned b = __float_as_uint(x);
    const int ex = (int)((b >> 23) & 255);
    const unsigned mant = ex == 0 ? 0u : (b & 0x7FFFFFu) | 0x800000u;
    const int sh = ex - 150 + e;  // |x| = mant 2^(ex - 150)
    const long long v = sh >= 0 ? (long long)((unsigned long long)mant << (sh & 63))
                                : (long long)(((mant >> min(-sh - 1, 31)) + 1) >> 1);
    return (b >> 31) ? -v : v;
}

// The same for a positive normal x.
__device__ __forceinline__ long long fix_of_positive(float x, int e) {
    const unsigned b = __float_as_uint(x), mant = (b & 0x7FFFFFu) | 0x800000u;
    const int sh = (int)(b >> 23) - 150 + e;
    return sh >= 0 ? (long long)((unsigned long long)mant << (sh & 63))
                   : (long long)(((mant >> min(-sh - 1, 31)) + 1) >> 1);
}

// Float pairs: a value is hi + lo, |lo| near 2^-24 |hi| at most.  Knuth's two-sum and the
// FMA product error are error-free; every operation is rounded by itself (_rn), so nothing is
// contracted or reassociated.
// Two floats in one register pair: packed FP32 operations, the IEEE result in both halves for one issue
// slot.
typedef unsigned long long F2;
__device__ __forceinline__ F2 pair2(float x, float y) {
    F2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(x), "f"(y));
    return r;
}
__device__ __forceinline__ F2 pair2(float x) { return pair2(x, x); }
__device__ __forceinline__ float lo2(F2 a) { return __uint_as_float((unsigned)a); }
__device__ __forceinline__ float hi2(F2 a) { return __uint_as_float((unsigned)(a >> 32)); }
__device__ __forceinline__ F2 neg2(F2 a) { return a ^ 0x8000000080000000ull; }
__device__ __forceinline__ F2 add2(F2 a, F2 b) {
    F2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ F2 sub2(F2 a, F2 b) {
    F2 r;
    asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ F2 mul2(F2 a, F2 b) {
    F2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ F2 fma2(F2 a, F2 b, F2 c) {
    F2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ void two_sum2(F2 a, F2 b, F2& s, F2& e) {
    s = add2(a, b);
    const F2 bv = sub2(s, a);
    e = add2(sub2(a, sub2(s, bv)), sub2(b, bv));
}
// The same where |a| >= |b| (Dekker's): half the operations.
__device__ __forceinline__ void fast_two_sum2(F2 a, F2 b, F2& s, F2& e) {
    s = add2(a, b);
    e = sub2(b, sub2(s, a));
}

// ln2/256 = kL0 + kL1 + kL2 (kL0 with 10 significant bits, so n kL0 is exact for n < 2^14;
// the three parts hold 58 bits) and 256/ln2.
constexpr float kL0 = 0x1.63p-9f, kL1 = -0x1.bd0106p-21f, kL2 = 0x1.cf79acp-48f;
constexpr float kInvL = 369.32993046757464f;

// k = exp(-|a - b|^2 / (2 l^2)) in the fixed point above, on the FP32 and integer pipes (the
// mixed-precision entries of the emulated kernel; the FP64 pipe is the scarce unit of the
// factorisation).  a, b: FP32 world coordinates (the inputs' own values), so each difference
// is exactly a float pair (two-sum) and |a - b|^2 is carried as a float pair renormalised
// after every axis;
//   y = |a - b|^2 / (2 l^2) as a float pair;
//   e^-y = 2^-(n/256) e^r with n = round(256 y / ln2) and r = n ln2/256 - y, |r| <= ln2/512
//   (Tang's table-driven reduction, as exp_neg), r as a normalised float pair, e^r from its
//   Taylor terms to r^4 (the next term is below 2^-54), 2^(i/256) from the float-pair table;
//   the float-pair result scaled by 2^(61 - m) into a 64-bit integer.
// The error stays below 2^-45 k (1 + y) + 2 units of 2^-61, about 2^-47 at most in k, at the
// level of the Cholesky's own backward error; 0 where y > 43.5 (k < 2^-62).  Bound by issue slots
// (about 110 FP32 and 40 integer operations an entry): two entries (b, b + 3) at once in packed FP32, and no
// error term where a sum is exact or ordered (2.5M queries of a city: 154.8 -> 150.9 ms in all,
// 152.2 of it without the packing).
__device__ __forceinline__ void kfix_ff2(const F2 (&a)[3], const float* b, F2 ch, F2 cl, const float2* tab,
                                         long long& k0, long long& k1) {
    F2 S, E;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const F2 nb = neg2(pair2(b[k], b[3 + k]));
        F2 dh, dl;
        two_sum2(a[k], nb, dh, dl);  // a - b = dh + dl exactly
        const F2 p = mul2(dh, dh), pe = fma2(dh, dh, neg2(p));
        // (dh + dl)^2 = p + pe + dl (2 dh + dl); then renormalise (S, E)
        const F2 rest = fma2(dl, fma2(pair2(2.f), dh, dl), pe);
        F2 t = p;
        if (k == 0) {
            E = rest;
        } else {
            F2 te;
            two_sum2(S, p, t, te);
            E = add2(E, add2(te, rest));
        }
        fast_two_sum2(t, E, S, E);
    }
    const F2 yh = mul2(S, ch);
    const F2 yl = add2(fma2(S, ch, neg2(yh)), fma2(S, cl, mul2(E, ch)));
    // (no branch on yh > 43.5: the entries of a strip then run interleaved)
    const F2 yn = mul2(yh, pair2(kInvL));
    const float n0 = rintf(lo2(yn)), n1 = rintf(hi2(yn));
    const F2 n = pair2(n0, n1);
    // r = (n kL0 - yh) + n kL1 - yl + n kL2, the large parts summed error-free.  n kL0 - yh is exact:
    // within a factor of two of each other from n = 2 (Sterbenz), and for n = 1 a multiple of 2^-33
    // below 2^-9.
    F2 b0, be, rh, ce;
    const F2 a0 = sub2(mul2(n, pair2(kL0)), yh);
    const F2 p2 = mul2(n, pair2(kL1)), p2e = fma2(n, pair2(kL1), neg2(p2));
    two_sum2(a0, p2, b0, be);
    two_sum2(b0, neg2(yl), rh, ce);
    const F2 rl = add2(add2(be, ce), fma2(n, pair2(kL2), p2e));
    // e^r - 1 = rh + rh^2/2 + [rl + rh rl + rh^3/6 + rh^4/24 + (rh^2 error)/2]
    const F2 q = mul2(rh, rh), qe = fma2(rh, rh, neg2(q));
    const F2 c34 = mul2(mul2(q, rh), fma2(rh, pair2(1.f / 24.f), pair2(1.f / 6.f)));
    const F2 small = add2(fma2(pair2(0.5f), qe, rl), fma2(rh, rl, c34));
    F2 u, ue, eh, e4;
    fast_two_sum2(rh, mul2(pair2(0.5f), q), u, ue);
    fast_two_sum2(pair2(1.f), u, eh, e4);
    const F2 el = add2(e4, add2(ue, small));
    // 2^(-n/256) = 2^-m 2^(i/256) with m = ceil(n / 256) and i = (-n) mod 256
    const int i0 = (int)n0, i1 = (int)n1;
    const int m0 = (i0 + 255) >> 8, m1 = (i1 + 255) >> 8;
    const float2 T0 = tab[-i0 & 255], T1 = tab[-i1 & 255];
    const F2 Tx = pair2(T0.x, T1.x), Ty = pair2(T0.y, T1.y);
    const F2 vh = mul2(Tx, eh);
    const F2 vl = add2(fma2(Tx, eh, neg2(vh)), fma2(Tx, el, mul2(Ty, eh)));
    k0 = lo2(yh) <= 43.5f ? fix_of_positive(lo2(vh), kFixBits - m0) + fix_of_float(lo2(vl), kFixBits - m0) : 0;
    k1 = hi2(yh) <= 43.5f ? fix_of_positive(hi2(vh), kFixBits - m1) + fix_of_float(hi2(vl), kFixBits - m1) : 0;
}

// The float pair (hi, lo) of an FP64 value.
__device__ __forceinline__ void split_pair(double v, float& hi, float& lo) {
    hi = (float)v;
    lo = (float)(v - (double)hi);
}

// Solve (L L^T) x = rhs in place on s.z (x written to out), L tile-packed; rows >= N of rhs
// must be zero.  Right-looking by 8-row blocks on each side.
__device__ void chol_solve(const Shared& s, const double* A, int Nt, double* out) {
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5, nwarps = nt >> 5;
    const int Np = Nt * 8;
    double* z = s.z;
    for (int kt = 0; kt < Nt; ++kt) {
        if (warp == (int)((kt + blockIdx.x) % nwarps)) {  // row r final, then out of the rows below it
            const double* D = A + tix(kt, kt);
            double v = lane < 8 ? z[8 * kt + lane] : 0.0;
            double d[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) d[r] = D[te(lane & 7, r)];
            const double inv = s.invd[8 * kt + (lane & 7)];
#pragma unroll
            for (int r = 0; r < 8; ++r) {
                if (lane == r) v *= inv;
                const double zr = __shfl_sync(0xffffffffu, v, r);
                if (lane > r) v = fma(-d[r], zr, v);
            }
            if (lane < 8) z[8 * kt + lane] = v;
        }
        __syncthreads();
        for (int i = 8 * (kt + 1) + tid; i < Np; i += nt) {
            const double* T = A + tix(i >> 3, kt);
            const int r = i & 7;
            double v = z[i];
#pragma unroll
            for (int c2 = 0; c2 < 8; ++c2) v -= T[te(r, c2)] * z[8 * kt + c2];
            z[i] = v;
        }
        __syncthreads();
    }
    for (int kt = Nt - 1; kt >= 0; --kt) {
        if (tid == 32 * (int)((kt + blockIdx.x) % nwarps)) {
            const double* D = A + tix(kt, kt);
#pragma unroll
            for (int r = 7; r >= 0; --r) {
                double v = z[8 * kt + r];
#pragma unroll
                for (int c2 = r + 1; c2 < 8; ++c2) v -= D[te(c2, r)] * out[8 * kt + c2];
                out[8 * kt + r] = v * s.invd[8 * kt + r];
            }
        }
        __syncthreads();
        for (int j = tid; j < 8 * kt; j += nt) {
            const double* T = A + tix(kt, j >> 3);
            const int cj = j & 7;
            double v = z[j];
#pragma unroll
            for (int c2 = 0; c2 < 8; ++c2) v -= T[te(c2, cj)] * out[8 * kt + c2];
            z[j] = v;
        }
        __syncthreads();
    }
}

// Start copying the tiles of the group of tile rows B0 .. B1 - 1 (at most kEB) that a solve takes one
// after the other into shared memory: the off-diagonal tiles (packed strict lower triangle), then
// the inverses of the diagonal tiles.  Thread i of n; complete after cp_async_wait and a barrier.
__device__ __forceinline__ double* solve_inverse(double* D, int k) { return D + (kDiagTiles - kEB + k) * 64; }
__device__ __forceinline__ double* solve_tile(double* D, int i, int j) { return D + (i * (i - 1) / 2 + j) * 64; }
__device__ __forceinline__ void cp_async_wait() { asm volatile("cp.async.wait_all;" ::: "memory"); }
__device__ __forceinline__ void load_solve_tiles(double* D, const double* A, const double* Tall, int B0, int B1, int i,
                                                 int n) {
    const int nb = B1 - B0;
    for (int x = i; x < nb * (nb + 1) / 2 * 32; x += n) {
        const int p = x >> 5, ir = tri_row(p), jc = p - ir * (ir + 1) / 2;
        const double* src = jc < ir ? A + eix(B0 + ir, B0 + jc) : Tall + 64 * (B0 + ir);
        double* dst = jc < ir ? solve_tile(D, ir, jc) : solve_inverse(D, ir);
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"((uint32_t)__cvta_generic_to_shared(dst + 2 * (x & 31))),
                     "l"(src + 2 * (x & 31))
                     : "memory");
    }
}

// Solve (L L^T) x = rhs in place on z (x written to out) with the inverses of every diagonal
// tile in Tall ([Nt][64], tile layout); rows >= N of rhs must be zero.  Groups of four tiles, one
// barrier per group and side.  A group's own solve is one dependent chain (64 FP64 operations of
// about 73 clocks, and 32 more for the previous group's part of its rows), so warp 0 does only that,
// from shared memory and from a row of 32 values loaded a group ahead, while the other warps take
// the previous group's solution out of the rows beyond and load the next group's tiles.  Every
// entry's operations keep one order: group by group, tile by tile.
__device__ __noinline__ void chol_solve_inv(double* z, double* Dsol, const double* A, int Nt, double* out,
                                            const double* Tall) {
    const int tid = threadIdx.x, nt = blockDim.x, lane = tid & 31, warp = tid >> 5;
    const int Np = Nt * 8;
    double row[4 * 8];  // warp 0: this lane's row (column) of the tiles that meet the previous group
    load_solve_tiles(Dsol, A, Tall, 0, min(kEB, Nt), tid, nt);
    cp_async_wait();
    __syncthreads();
    for (int B0 = 0, par = 0; B0 < Nt; B0 += kEB, par ^= 1) {  // L y = rhs
        const int B1 = min(B0 + kEB, Nt);
        double* D = Dsol + par * kDiagTiles * 64;
        if (warp == 0) {
            const int i = 8 * B0 + lane;  // the group's rows less the previous group's part
            if (B0 > 0 && i < 8 * B1) {
                double u = z[i];
#pragma unroll
                for (int e = 0; e < 32; ++e) u -= row[e] * z[8 * (B0 - kEB) + e];
                z[i] = u;
            }
            const int in = 8 * B1 + lane;
            if (in < Np) {
#pragma unroll
                for (int e = 0; e < 32; e += 2) {
                    const double2 v = *reinterpret_cast<const double2*>(A + eix(in >> 3, B0 + (e >> 3)) + te(in & 7, e & 7));
                    row[e] = v.x;
                    row[e + 1] = v.y;
                }
            }
            __syncwarp();
            for (int k = 0; k < B1 - B0; ++k) {
                const double* Ti = solve_inverse(D, k);
                double* zk = z + 8 * (B0 + k);
                double v = 0.0;
                if (lane < 8)
#pragma unroll
                    for (int c2 = 0; c2 < 8; ++c2)
                        if (c2 <= lane) v += Ti[te(lane, c2)] * zk[c2];
                __syncwarp();
                if (lane < 8) zk[lane] = v;
                __syncwarp();
                const int il = 8 * (k + 1) + lane;  // rows of the group below tile k
                if (il < 8 * (B1 - B0)) {
                    const double* T = solve_tile(D, il >> 3, k);
                    const int r = il & 7;
                    double u = z[8 * B0 + il];
#pragma unroll
                    for (int c2 = 0; c2 < 8; ++c2) u -= T[te(r, c2)] * zk[c2];
                    z[8 * B0 + il] = u;
                }
                __syncwarp();
            }
        } else {
            if (B1 < Nt)
                load_solve_tiles(Dsol + (par ^ 1) * kDiagTiles * 64, A, Tall, B1, min(B1 + kEB, Nt), tid - 32, nt - 32);
            if (B0 > 0)
                for (int i = 8 * B1 + tid - 32; i < Np; i += nt - 32) {
                    const int r = i & 7;
                    double u = z[i];
#pragma unroll
                    for (int k = 0; k < kEB; ++k) {
                        const double* T = A + eix(i >> 3, B0 - kEB + k);
                        const double* zk = z + 8 * (B0 - kEB + k);
#pragma unroll
                        for (int c2 = 0; c2 < 8; ++c2) u -= T[te(r, c2)] * zk[c2];
                    }
                    z[i] = u;
                }
            cp_async_wait();
        }
        __syncthreads();
    }
    // L^T x = y, groups of kEB tiles from the last tile on
    load_solve_tiles(Dsol, A, Tall, max(Nt - kEB, 0), Nt, tid, nt);
    cp_async_wait();
    __syncthreads();
    for (int B1 = Nt, par = 0; B1 > 0; B1 -= kEB, par ^= 1) {
        const int B0 = max(B1 - kEB, 0);
        double* D = Dsol + par * kDiagTiles * 64;
        if (warp == 0) {
            const int j = 8 * B0 + lane;  // the group's columns less the next group's part
            if (B1 < Nt && j < 8 * B1) {
                double u = z[j];
#pragma unroll
                for (int e = 0; e < 32; ++e) u -= row[e] * out[8 * B1 + e];
                z[j] = u;
            }
            // for the group before: the columns of its tiles that meet this (full) group
            const int P0 = max(B0 - kEB, 0), jn = 8 * P0 + lane;
            if (jn < 8 * B0) {
#pragma unroll
                for (int e = 0; e < 32; ++e) row[e] = A[eix(B0 + (e >> 3), jn >> 3) + te(e & 7, jn & 7)];
            }
            __syncwarp();
            for (int k = B1 - B0 - 1; k >= 0; --k) {
                const double* Ti = solve_inverse(D, k);
                const int kt = B0 + k;
                double v = 0.0;
                if (lane < 8)
#pragma unroll
                    for (int r = 0; r < 8; ++r)
                        if (r >= lane) v += Ti[te(r, lane)] * z[8 * kt + r];
                __syncwarp();
                if (lane < 8) out[8 * kt + lane] = v;
                __syncwarp();
                if (lane < 8 * k) {  // columns of the group left of tile k
                    const double* T = solve_tile(D, k, lane >> 3);
                    const int cj = lane & 7;
                    double u = z[8 * B0 + lane];
#pragma unroll
                    for (int c2 = 0; c2 < 8; ++c2) u -= T[te(c2, cj)] * out[8 * kt + c2];
                    z[8 * B0 + lane] = u;
                }
                __syncwarp();
            }
        } else {
            if (B0 > 0)
                load_solve_tiles(Dsol + (par ^ 1) * kDiagTiles * 64, A, Tall, max(B0 - kEB, 0), B0, tid - 32, nt - 32);
            if (B1 < Nt)
                for (int j = tid - 32; j < 8 * B0; j += nt - 32) {
                    const int cj = j & 7;
                    double u = z[j];
#pragma unroll
                    for (int k = 0; k < kEB; ++k) {
                        const double* T = A + eix(B1 + k, j >> 3);
                        const double* ok = out + 8 * (B1 + k);
#pragma unroll
                        for (int c2 = 0; c2 < 8; ++c2) u -= T[te(c2, cj)] * ok[c2];
                    }
                    z[j] = u;
                }
            cp_async_wait();
        }
        __syncthreads();
    }
}

// Which entry of the update of step j (below) a lane takes: its place in the tile (bits 0-5; bit 6: in
// T, else in S), or 128 for none.
__device__ __forceinline__ uint8_t diag_entry(int j, int lane) {
    const int m = 7 - j, nc = m * (m + 1) / 2;  // pairs of rows of S, then rows and columns of T
    if (lane >= nc + m * (j + 1)) return 128;
    if (lane < nc) {
        const int a = tri_row(lane);
        return (uint8_t)te(j + 1 + a, j + 1 + lane - a * (a + 1) / 2);
    }
    const int q = lane - nc;
    return (uint8_t)(te(j + 1 + q / (j + 1), q % (j + 1)) | 64);
}

// One warp: the 8x8 Cholesky of the diagonal tile S in place (lower part), 1 / L_jj into invd, and the
// inverse of its factor into T (upper part zero).  One pass over the tile and the identity beside
// it: step j scales column j of S and row j of T by 1 / L_jj in one operation and takes their
// products out of the rows below in one more (two where they are over 32).  An FP64 operation
// holds its sub-partition for about 66 clocks however few lanes are on, so what counts is their
// number: about 8 a step with kRsqrt, 17 without, and none for the inverse by itself.  On one
// thread, entry by entry, a tile took about 400.  kRsqrt: 1 / L_jj from rsqrt (emulated kernel), else
// 1 / sqrt.  tab: diag_entry of every step and lane.  False on a non-positive pivot (the same on every lane).
template <bool kRsqrt>
__device__ __forceinline__ bool diag_tile_warp(double* S, double* T, double* invd, const uint8_t* tab) {
    const int lane = threadIdx.x & 31;
    T[lane] = 0.0;
    T[lane + 32] = 0.0;
    __syncwarp();
#pragma unroll 1
    for (int j = 0; j < 8; ++j) {
        const int e = tab[32 * j + lane], row = (e >> 3) & 7, col = (e & 7) ^ ((row & 2) << 1);
        double* const M = e & 64 ? T : S;
        const int f1 = te(row, j), f2 = e & 64 ? te(j, col) : te(col, j);
        // the lane's entry of the scaling: S_ij for lanes i = j .. 7, T_jc for lanes 8 + c, c <= j
        double* const xs = lane < 8 ? S + te(lane, j) : T + te(j, lane & 7);
        const bool on = lane < 8 ? lane >= j : lane <= 8 + j;
        const double v = S[te(j, j)];
        double x = on ? *xs : 0.0;
        if (lane == 8 + j) x = 1.0;
        if (!(v > 0.0)) return false;
        double r, y;
        if (kRsqrt) {
            r = rsqrt(v);
            y = x * r;
        } else {
            const double d = sqrt(v);
            r = 1.0 / d;
            y = x * r;
            if (lane == j) y = d;
        }
        __syncwarp();
        if (on) *xs = y;
        if (lane == 0) invd[j] = r;
        __syncwarp();
        if (e < 128) M[e & 63] -= S[f1] * M[f2];
        if (j < 2 && lane < 3 - 2 * j) {  // the entries of T beyond 32: (5 .. 7, 0) and (7, 1)
            const int r2 = j == 0 ? 5 + lane : 7;
            T[te(r2, j)] -= S[te(r2, j)] * T[te(j, j)];
        }
        __syncwarp();
    }
    return true;
}

// w 2^sh rounded to an integer (ties up) for a 64-bit integer w: a slice-product update in
// the fixed point of the trailing matrix.  No overflow: |w| 2^sh is bounded by the entry bound.
__device__ __forceinline__ long long fix_shift(long long w, int sh) {
    const int n = min(-sh - 1, 63);  // a shift by 63 leaves -1 or 0, which rounds to 0
    return sh >= 0 ? w << sh : ((w >> (n & 63)) + 1) >> 1;
}

// The update w of an entry from its eight slice groups (see factor_emulated), given as the bits of
// G + 1.5 * 2^23 (kGroupBits + G, exact for |G| < 2^22):
//   w = 2^40 G_0 + 2^32 G_1 + ... + 2^16 G_3 + round((2^24 G_4 + 2^16 G_5 + 2^8 G_6 + G_7) / 2^16),
// pairs of groups joined in 32 bits first (|256 G + G'| < 2^31), so the 64-bit part is one wide
// multiply-add and one addition to the high word.
constexpr unsigned kGroupBits = 0x4B400000u;
static_assert(7 * 8 * kEB * 128 * 128 < 1 << 22, "a slice group of a block's columns exceeds 22 bits");
__device__ __forceinline__ long long join_groups(const unsigned (&g)[8]) {
    constexpr unsigned kOff = kGroupBits * 257u;
    const unsigned a = g[0] * 256u + g[1] - kOff;
    const int b = (int)(g[2] * 256u + g[3] - kOff);
    const unsigned c = g[4] * 256u + g[5] - kOff;
    const int d = (int)(g[6] * 256u + g[7] - kOff + 32768u);
    const int e = (int)(c + (unsigned)(d >> 16));
    return (long long)b * 65536 + e + (long long)((unsigned long long)a << 32);
}

// Balanced base-256 digits of row g of an 8-row tile over one block (the FP64 values
// x[0 .. 2 kEB - 1] held by the four lanes t of the row: columns 8 j + 2t and 8 j + 2t + 1 in
// x[2j], x[2j + 1]), written as bf16 pairs to F (slices kColT kSliceBytes apart) in the tensor cores'
// K-major layout: [core matrix of 8 columns][row][8 bf16], 16 bytes per row and 128 per core
// matrix; and the row scale 2^(em - 1021) to *scale (lane t = 0).  The digit scheme is described at factor_emulated.
// With u (an appended query row's diagonal entry in the fixed point, lane t = 0) the row's own
// update |row|^2 is taken from the digits here: only the diagonal of the query-by-query block is
// needed, and 19 integer products per column cost a tenth of the tensor-core tiles that hold it.
__device__ __forceinline__ void slice_row(const double (&x)[2 * kEB], uint32_t* F, double* scale, long long* u) {
    const int lane = threadIdx.x & 31;
    int em = 0;
#pragma unroll
    for (int i = 0; i < 2 * kEB; ++i) em = max(em, (int)((__double_as_longlong(x[i]) >> 52) & 0x7FF));
    em = max(em, __shfl_xor_sync(0xffffffffu, em, 1));
    em = max(em, __shfl_xor_sync(0xffffffffu, em, 2));
    unsigned G[8] = {0, 0, 0, 0, 0, 0, 0, 0};
#pragma unroll
    for (int kk = 0; kk < kEK; ++kk) {
        unsigned long long Yb[4];
        bool negx[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {  // columns 16 kk + {2t, 2t + 1, 8 + 2t, 8 + 2t + 1}
            const unsigned long long bits = (unsigned long long)__double_as_longlong(x[4 * kk + i]);
            const int E = (int)((bits >> 52) & 0x7FF);
            unsigned long long Y = 0;  // |x| 2^(1077 - em) rounded to nearest, below 2^55
            if (E > 0 && E < 0x7FF) {  // zero and subnormals slice to zero
                const int sh = em - E;
                const unsigned long long M = ((bits & 0xFFFFFFFFFFFFFull) | (1ull << 52)) << 2;
                Y = sh == 0 ? M : sh >= 56 ? 0ull : ((M >> (sh - 1)) + 1) >> 1;
            }
            // adding 128 to each of the six lower digits lets every digit be read as a byte
            // minus 128; the top digit keeps the rest (0 .. 128)
            Yb[i] = Y + 0x808080808080ull;
            negx[i] = (bits >> 63) != 0;
        }
#pragma unroll
        for (int ss = 0; ss < 7; ++ss) {  // ss = 0: the most significant digit
            uint32_t h16[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                int qv = ss == 0 ? (int)(Yb[i] >> 48) : (int)((Yb[i] >> (48 - 8 * ss)) & 255ull) - 128;
                if (negx[i]) qv = -qv;
                h16[i] = __float_as_uint((float)qv) >> 16;  // exact: |qv| <= 2^7
            }
            // lane = 4 g + t: row g, columns 2t, 2t + 1 of the core matrices of columns 0-7 and 8-15
            F[ss * (kColT * kSliceBytes / 4) + kk * 64 + lane] = h16[0] | (h16[1] << 16);
            F[ss * (kColT * kSliceBytes / 4) + kk * 64 + 32 + lane] = h16[2] | (h16[3] << 16);
        }
        if (u) {  // G_g += sum_{s+t=g} q_s q_t of each column (the sign drops out)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                int q[7];
                q[0] = (int)(Yb[i] >> 48);
#pragma unroll
                for (int ss = 1; ss < 7; ++ss) q[ss] = (int)((Yb[i] >> (48 - 8 * ss)) & 255ull) - 128;
#pragma unroll
                for (int gq = 0; gq < 8; ++gq) {
                    int v = 0;
#pragma unroll
                    for (int ss = 0; 2 * ss < gq; ++ss)
                        if (gq - ss < 7) v += q[ss] * q[gq - ss];
                    v *= 2;
                    if (gq % 2 == 0) v += q[gq / 2] * q[gq / 2];
                    G[gq] += (unsigned)v;
                }
            }
        }
    }
    if ((lane & 3) == 0) *scale = em > 0 ? __longlong_as_double((long long)(em + 2) << 52) : 0.0;
    if (u) {
#pragma unroll
        for (int gq = 0; gq < 8; ++gq) {
            G[gq] += __shfl_xor_sync(0xffffffffu, G[gq], 1);
            G[gq] += __shfl_xor_sync(0xffffffffu, G[gq], 2);
            G[gq] += kGroupBits;
        }
        const int e = em > 0 ? em + 2 : 0;
        if ((lane & 3) == 0) *u -= fix_shift(join_groups(G), 2 * e - (2102 - kFixBits));
    }
}

// acc_i -= x_0 l_i0 + ... + x_7 l_i7 for the two columns i = c0, c1 of tile L and the row X points at
// (r: its row in the tile), one operation after the other in that order.
__device__ __forceinline__ void sub_products(double& acc0, double& acc1, const double* X, int r, const double* L, int c0,
                                             int c1) {
#pragma unroll
    for (int m = 0; m < 8; m += 2) {
        const double2 x = *reinterpret_cast<const double2*>(X + te(r, m));
        const double2 u = *reinterpret_cast<const double2*>(L + te(c0, m));
        const double2 v = *reinterpret_cast<const double2*>(L + te(c1, m));
        acc0 = fma(-x.x, u.x, acc0);
        acc1 = fma(-x.x, v.x, acc1);
        acc0 = fma(-x.y, u.y, acc0);
        acc1 = fma(-x.y, v.y, acc1);
    }
}

// The row r of a tile P times Ti^T, columns c0 <= 3 and c1 (Ti lower triangular, its upper part zero).
__device__ __forceinline__ void times_inverse(double& y0, double& y1, const double* P, int r, const double* Ti, int c0,
                                              int c1) {
    y0 = y1 = 0.0;
#pragma unroll
    for (int m = 0; m < 8; m += 2) {
        const double2 p = *reinterpret_cast<const double2*>(P + te(r, m));
        const double2 v = *reinterpret_cast<const double2*>(Ti + te(c1, m));
        if (m < 4) {
            const double2 u = *reinterpret_cast<const double2*>(Ti + te(c0, m));
            y0 = fma(p.x, u.x, y0);
            y0 = fma(p.y, u.y, y0);
        }
        y1 = fma(p.x, v.x, y1);
        y1 = fma(p.y, v.y, y1);
    }
}

// Row tile it below the factorised diagonal block of tile columns K0 .. K0 + kEB - 1 (its tiles in
// Dblk, the inverses of its diagonal tiles in Tblk): L_it,K0+j = (A_it,K0+j - sum_{k<j} L_it,K0+k L_K0+j,K0+k^T)
// Ti_j^T for j < kEB, one warp, lane = 4 g + t: row g, columns t and 7 - t of each tile (so that the
// zeros of Ti cost the same on every lane).  W: kEB tiles of scratch, the solved tiles.  The
// results are stored to A and sliced for the trailing update (F, scale: this tile's slices
// and row scales; u: the diagonal entries of an appended query tile's rows, else null).
// Bound by the FP64 pipe: 144 operations of 66 clocks.  As 8x8x4 FP64 MMAs (the same chain of fused
// multiply-adds, bit for bit) it was 20 of 580 clocks, zeros of Ti included.
__device__ void block_rows(double* A, int it, int K0, const double* Dblk, const double* Tblk, double* W,
                           uint32_t* F, double* scale, long long* u) {
    const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
    double* R = A + eix(it, K0);  // tiles (it, K0 .. K0 + kEB - 1), kTileCol apart
    double a0[kEB], a1[kEB];
#pragma unroll
    for (int j = 0; j < kEB; ++j) {
        a0[j] = R[kTileCol * j + te(g, t)];
        a1[j] = R[kTileCol * j + te(g, 7 - t)];
    }
#pragma unroll
    for (int j = 0; j < kEB; ++j) {
        const double* Lj = Dblk + j * (j + 1) / 2 * 64;  // tiles (K0 + j, K0 .. K0 + j)
#pragma unroll
        for (int k = 0; k < j; ++k) sub_products(a0[j], a1[j], W + 64 * k, g, Lj + 64 * k, t, 7 - t);
        double* Wj = W + 64 * j;
        Wj[te(g, t)] = a0[j];
        Wj[te(g, 7 - t)] = a1[j];
        __syncwarp();
        double y0, y1;
        times_inverse(y0, y1, Wj, g, Tblk + 64 * j, t, 7 - t);
        __syncwarp();
        Wj[te(g, t)] = y0;
        Wj[te(g, 7 - t)] = y1;
        __syncwarp();
    }
    double x[2 * kEB];  // columns 2t, 2t + 1 of each tile
#pragma unroll
    for (int j = 0; j < kEB; ++j) {
        const double2 v = *reinterpret_cast<const double2*>(W + 64 * j + te(g, 2 * t));
        *reinterpret_cast<double2*>(R + kTileCol * j + te(g, 2 * t)) = v;
        x[2 * j] = v.x;
        x[2 * j + 1] = v.y;
    }
    __syncwarp();
    slice_row(x, F, scale + g, u ? u + g : nullptr);
}

// Workspace of the emulated factorisation, per CTA or cluster: the slices of the rows below the current block
// ([group of 4 row tiles][slice][row tile][4 core matrices], 3584 bytes per row tile), the row scales, the inverses of
// all diagonal tiles ([rows / 8][64] doubles), and the appended query rows' diagonal entries in
// the fixed point.
__device__ __forceinline__ unsigned char* emu_ws(const SolveCtx& c) { return c.ws_e + (int64_t)(blockIdx.x / c.ncta) * c.ws_e_stride; }
__device__ __forceinline__ int emu_rows(const SolveCtx& c) { return c.nrow > 0 ? c.nrow : c.npad; }
__device__ __forceinline__ double* emu_scales(const SolveCtx& c) {
    return reinterpret_cast<double*>(emu_ws(c) + (int64_t)(emu_rows(c) / 8) * kSliceTileBytes);
}
__device__ __forceinline__ double* emu_tile_inverses(const SolveCtx& c) { return emu_scales(c) + emu_rows(c); }
__device__ __forceinline__ long long* emu_query_diag(const SolveCtx& c) {
    return reinterpret_cast<long long*>(emu_tile_inverses(c) + 8 * emu_rows(c));
}

// ---- tensor-core (tcgen05) helpers for the emulated updates --------------------------------
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory matrix descriptor, K-major without swizzle: core matrices of 8 rows x 16 bytes,
// the next along K lbo bytes on, the next along M or N sbo bytes on.
__device__ __forceinline__ uint64_t umma_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
    return (uint64_t)((saddr >> 4) & 0x3FFF) | ((uint64_t)((lbo >> 4) & 0x3FFF) << 16) |
           ((uint64_t)((sbo >> 4) & 0x3FFF) << 32) | (1ull << 46);
}

// Instruction descriptor of kind::f16: bf16 A and B (K-major), FP32 D, M = 128, N = n.
__host__ __device__ constexpr uint32_t umma_idesc(int n) {
    return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n / 8) << 17) | ((uint32_t)(128 / 16) << 24);
}

__device__ __forceinline__ void umma_bf16(uint32_t d_tmem, uint64_t a, uint64_t b, int n, uint32_t accumulate) {
    asm volatile("{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
                 " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}"
                 ::"r"(d_tmem), "l"(a), "l"(b), "r"(umma_idesc(n)), "r"(accumulate));
}

__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint32_t bar) {
    asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
                 ::"r"(smem_addr(dst)), "l"(src), "r"(bytes), "r"(bar) : "memory");
}

// Wait of the calling thread for the completion of phase `parity` of an mbarrier, at most
// kWaitLimit polls (false: the wait gave up).
constexpr int kWaitLimit = 1 << 18;
__device__ __forceinline__ bool bar_poll(uint32_t bar, uint32_t parity) {
    uint32_t done = 0;
    for (int it = 0; it < kWaitLimit && !done; ++it)
        asm volatile("{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
                     " selp.u32 %0, 1, 0, p;\n}"
                     : "=r"(done) : "r"(bar), "r"(parity) : "memory");
    return done != 0;
}
// The same for the whole CTA: the result is the same on every thread.
__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity) {
    return __syncthreads_and((int)bar_poll(bar, parity)) != 0;
}

// Tensor memory and barriers of an emulated CTA.  kGroup: several CTAs (a cluster) work on one instance
// together; without it they are one, known to the compiler (1 to 7 % faster for the large batches).
template <bool kGroup>
struct EmuTc {
    uint32_t tmem;       // base of kEmuTmemCols columns: slice group g at columns 8 kColT g
    uint32_t bar_ld;     // completion of the staging copies
    uint32_t bar_mma;    // completion of the MMAs
    uint32_t ph_ld, ph_mma;
    bool dead;           // a bounded wait gave up: take no more work
    // the CTAs that work together: how many, this one's rank, and two sets of shared-memory words,
    // one for each rank's flag
    int n_, rank_;
    int* flags;
    int set;
    __device__ __forceinline__ int n() const { return kGroup ? n_ : 1; }
    __device__ __forceinline__ int rank() const { return kGroup ? rank_ : 0; }
};

// The shared-memory word of the cluster's CTA `rank` that lies where p does in this one.
__device__ __forceinline__ uint32_t peer_word(const void* p, int rank) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_addr(p)), "r"(rank));
    return a;
}
__device__ __forceinline__ void peer_store(const void* p, int rank, int v) {
    asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(peer_word(p, rank)), "r"(v) : "memory");
}

// Barrier of the CTAs that work together (of this CTA alone without a cluster): what any of them wrote
// before it is seen by all after it.  Returns whether any thread passed a flag, the same everywhere:
// each CTA leaves its own in every other's words before it arrives; the two sets alternate, so
// a word is written again only after everyone has read it.
template <class Tc>
__device__ __forceinline__ bool group_sync(Tc& tc, int flag) {
    const int any = __syncthreads_or(flag);
    if (tc.n() == 1) return any != 0;
    int* f = tc.flags + 8 * tc.set;
    if ((int)threadIdx.x < tc.n()) peer_store(f + tc.rank(), threadIdx.x, any);
    __syncwarp();  // (the aligned barrier wants the whole warp, and only its first lanes stored)
    asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
    asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
    int all = 0;
    for (int i = 0; i < tc.n(); ++i) all |= reinterpret_cast<volatile int*>(f)[i];
    tc.set ^= 1;
    return all != 0;
}
template <class Tc>
__device__ __forceinline__ void group_barrier(Tc& tc) {
    if (tc.n() == 1)
        __syncthreads();
    else
        group_sync(tc, 0);
}

// columns a tensor-memory load reads for each lane (four, with nothing else in flight: 154.8 ms for the
// city step; two at a time with the next two in flight 157.0, eight 154.8 with more spills)
constexpr int kLdCols = 4;
__device__ __forceinline__ void tmem_ld(uint32_t taddr, uint32_t (&v)[kLdCols]) {
    asm volatile("tcgen05.ld.sync.aligned.32x32b.x4.b32 {%0,%1,%2,%3}, [%4];"
                 : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]) : "r"(taddr) : "memory");
}
// The loaded values pass through the wait, so no use of them is scheduled before it.
__device__ __forceinline__ void tmem_wait_ld(uint32_t (&v)[8][kLdCols]) {
    asm volatile("tcgen05.wait::ld.sync.aligned;" : : : "memory");
#pragma unroll
    for (int g = 0; g < 8; ++g)
#pragma unroll
        for (int e = 0; e < kLdCols; ++e) asm volatile("" : "+r"(v[g][e]));
}

// A bounded wait gave up: record it; the CTA stops taking work.
template <class Tc>
__device__ __forceinline__ bool emu_fail(const SolveCtx& c, Tc& tc) {
    if (threadIdx.x == 0) atomicOr(c.err, kErrTimeout);
    tc.dead = true;
    return false;
}

// Trailing update C -= P P^T of the M = Nt - K1 row tiles below the block that ends at K1, on
// the tensor cores, for the columns of the matrix itself (row tiles K1 .. Ntr - 1).  P's rows are
// cut into seven digit slices (see factor_emulated), and every slice group
// G_g = sum_{s+t=g} P_s P_t^T is accumulated exactly in FP32 in tensor memory.  Output tiles of
// kBandT row tiles (128 rows) by kColT row tiles (32 columns) cover the lower triangle, band by
// band.  Bulk copies stage the band's slices (A) once per band and each column tile's slices (B)
// in one of two buffers, the next tile's while the current one computes.
//
// The groups lie side by side in tensor memory (group g at columns 32 g) and B's slices side by
// side in shared memory, so A slice s times B slices 0 .. n - 1 is ONE product of N = 32 n columns
// whose output lands on groups s .. s + n - 1: 15 MMAs per tile instead of 68 of N = 32, each
// reading its 4 KB of A from shared memory once.  An N = 32 product is bound by that read (about
// 40 clocks for 16 of arithmetic); all of a tile's now need about 1100 clocks, the arithmetic's.
// One thread issues them.  All 8 warps then read their rows (lane quadrant warp % 4) and columns
// (half warp / 4) of the groups, join each element's groups into one integer and subtract it from
// the fixed point.  C is read and written in whole 256-byte lines (see bix); the next tile's block
// is prefetched into L2.  Measured against 68 N = 32 products, 8-byte accesses to 64-byte tile rows
// and a diagonal of the query block from full tiles: 38 instances of about 790 points alone on the
// GPU 16.1 -> 11.7 ms, 15.6k of 4 to 1024 points 216 -> 180 ms.
// With a cluster the call takes the part's tiles r, r + n, .. of each band (r + 1, .. in the next band).
enum class TilePart { kAll, kFirst, kRest };  // kFirst: the first band's first tile, kRest: all but it
template <class Tc>
__device__ bool trailing_update_tc(double* A, int Nt, int Ntr, int K1, const unsigned char* E,
                                   const double* sr, unsigned char* stage, Tc& tc, int r, int n, TilePart part) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
    const int M = Nt - K1;
    const int jr = (max(Ntr - K1, 0) + kColT - 1) / kColT;  // column tiles
    auto tiles_of = [&](int b0) {
        if (part == TilePart::kFirst) return b0 == 0 ? 1 : 0;
        return min(jr, (b0 + min(kBandT, M - b0) + kColT - 1) / kColT);
    };
    auto first_of = [&](int b0) {
        const int f = (r + b0 / kBandT) % n;
        return part == TilePart::kRest && b0 == 0 && f == 0 ? n : f;
    };
    auto next_band = [&](int b0) {  // the first band from b0 on that has a tile for this CTA
        while (b0 < M && first_of(b0) >= tiles_of(b0)) b0 += kBandT;
        return b0;
    };
    int b0 = next_band(0);
    if (jr == 0 || b0 >= M) return true;
    const uint32_t aA = smem_addr(stage), aB = aA + kStageA;
    const int q = warp & 3, h = warp >> 2;  // lane quadrant (rows 32 q ..) and column half
    const int kb1 = K1 >> 2;                // 32-row block of the first row below (K1 is a multiple of 4)
    int fail = 0;
    // the band's A (warp w: slice w, a lane per group of 4 row tiles) and its first column tile's B
    // (buffer 0, warp 7, which also arms the barrier)
    auto stage_band = [&](int b0) {
        const int ng = (min(kBandT, M - b0) + kColT - 1) / kColT;
        const unsigned char* G = E + (int64_t)(b0 / kColT) * kGroupBytes;
        if (warp < 7) {
            if (lane < ng)
                bulk_load(stage + warp * (kStageA / 7) + lane * (kStageB / 7), G + (int64_t)lane * kGroupBytes + warp * (kStageB / 7),
                          kStageB / 7, tc.bar_ld);
        } else if (lane == 0) {
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(tc.bar_ld),
                         "r"((uint32_t)(ng + 1) * kGroupBytes)
                         : "memory");
            bulk_load(stage + kStageA, E + (int64_t)first_of(b0) * kGroupBytes, kStageB, tc.bar_ld);
        }
    };
    stage_band(b0);
    for (int b1; b0 < M; b0 = b1) {
        b1 = next_band(b0 + kBandT);
        const int nb = min(kBandT, M - b0);
        const int rb = (b0 >> 2) + q;              // the warp's 32-row block below K1
        const bool rows_in = 4 * q < nb;
        // the row's exponent (rows past the matrix inside its last block: unused)
        const int er = rows_in ? (int)(__double_as_longlong(sr[32 * rb + lane]) >> 52) : 0;
        const int n_tiles = tiles_of(b0);  // column tiles reaching the band's last row
        for (int jt = first_of(b0), buf = 0; jt < n_tiles; jt += n, buf ^= 1) {
            const uint32_t bufB = aB + (uint32_t)(buf * kStageB);
            // this thread's 16 entries of C (one row, 16 columns) and the column scales, all loads
            // issued at once; they arrive while the MMAs run
            const bool on = rows_in && jt <= rb;  // (warp-uniform, as the collective tcgen05.ld needs)
            long long* C = reinterpret_cast<long long*>(A + bix(kb1 + rb, kb1 + jt)) + 512 * h;
            long long cv[16];
            double es = 0.0;
            if (on) {
#pragma unroll
                for (int cc = 0; cc < 16; ++cc) cv[cc] = C[32 * cc + lane];
                es = sr[32 * jt + 16 * h + (lane & 15)];
                if (jt + n < n_tiles && jt + n <= rb && lane == 0)
                    asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(C + 1024 * n), "r"(4096));
            }
            // warp 0 alone waits for the copies, starts the next ones and issues the products: every
            // phase of the copy barrier is seen before the next one can start
            if (warp == 0 && !bar_poll(tc.bar_ld, tc.ph_ld)) fail = 1;
            if (warp == 0 && !__any_sync(0xffffffffu, fail) && lane == 0) {
                if (jt + n < n_tiles) {  // the next column tile's B into the other buffer
                    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(tc.bar_ld),
                                 "r"((uint32_t)kStageB)
                                 : "memory");
                    bulk_load(stage + kStageA + (buf ^ 1) * kStageB, E + (int64_t)(jt + n) * kGroupBytes, kStageB,
                              tc.bar_ld);
                }
                asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
                for (int kh = 0; kh < 2; ++kh)
#pragma unroll
                    for (int ss = 0; ss < 7; ++ss) {
                        const int n = ss == 0 ? 7 : 8 - ss;  // B slices of this product
                        const uint64_t da = umma_desc(aA + ss * (kStageA / 7) + kh * 256, 128, kSliceBytes);
                        const uint32_t b = bufB + kh * 256;
                        const uint32_t dcol = tc.tmem + ss * 8 * kColT;
                        if (kh == 0 && ss == 1) {
                            // groups 1 .. 6 hold slice 0's products; group 7 starts here
                            umma_bf16(dcol, da, umma_desc(b, 128, kSliceBytes), 6 * 8 * kColT, 1u);
                            umma_bf16(dcol + 6 * 8 * kColT, da, umma_desc(b + 6 * kColT * kSliceBytes, 128, kSliceBytes),
                                      8 * kColT, 0u);
                        } else {
                            umma_bf16(dcol, da, umma_desc(b, 128, kSliceBytes), n * 8 * kColT, (kh == 0 && ss == 0) ? 0u : 1u);
                        }
                    }
                asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(tc.bar_mma)
                             : "memory");
            }
            __syncwarp();
            tc.ph_ld ^= 1;
            const int ec_lane = (int)(__double_as_longlong(es) >> 52);
            if (!bar_poll(tc.bar_mma, tc.ph_mma)) fail = 1;
            tc.ph_mma ^= 1;
            __syncwarp();
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            // the band's last products are done (so warp 0 has seen every copy): its A and B buffers
            // take the next band's
            if (!__any_sync(0xffffffffu, fail) && jt + n >= n_tiles && b1 < M) {
                stage_band(b1);
                __syncwarp();  // (some lanes copied; the aligned tensor-memory loads want the whole warp)
            }
            if (on) {
                const uint32_t tbase = tc.tmem + ((uint32_t)(32 * q) << 16) + (uint32_t)(16 * h);
#pragma unroll
                for (int p = 0; p < 16 / kLdCols; ++p) {
                    uint32_t v[8][kLdCols];
#pragma unroll
                    for (int gq = 0; gq < 8; ++gq) tmem_ld(tbase + (uint32_t)(gq * 8 * kColT + kLdCols * p), v[gq]);
                    tmem_wait_ld(v);
#pragma unroll
                    for (int e = 0; e < kLdCols; ++e) {
                        unsigned gb[8];
#pragma unroll
                        for (int gq = 0; gq < 8; ++gq)
                            gb[gq] = __float_as_uint(__fadd_rn(__uint_as_float(v[gq][e]), 12582912.0f));
                        const int ec = __shfl_sync(0xffffffffu, ec_lane, kLdCols * p + e);
                        // the update is w 2^(er + ec - 2102), in units of 2^-kFixBits
                        cv[kLdCols * p + e] -= fix_shift(join_groups(gb), er + ec - (2102 - kFixBits));
                    }
                }
                // the next block's columns are final after this update: stored as FP64 tiles (see
                // factor_emulated), the rest in the fixed point.  The half block is read before it
                // is written in the other form.
                if (jt == 0) {
                    __syncwarp();
                    double* T = reinterpret_cast<double*>(C) + (lane >> 3) * 64;
                    const int rr = lane & 7;
#pragma unroll
                    for (int cc = 0; cc < 16; cc += 2)
                        *reinterpret_cast<double2*>(T + (cc >> 3) * kTileCol + te(rr, cc & 7)) =
                            make_double2(double_of_fix(cv[cc]), double_of_fix(cv[cc + 1]));
                } else {
#pragma unroll
                    for (int cc = 0; cc < 16; ++cc) C[32 * cc + lane] = cv[cc];
                }
            }
            // every thread's reads of the accumulators are done before the next tile's MMAs
            asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
            if (__syncthreads_or(fail)) return false;
        }
    }
    return true;
}

// Right-looking Cholesky of a global-memory instance in blocks of W = 8 kEB columns, with
// every trailing update C -= P P^T (P: the block's W columns below it) done on the bf16
// tensor cores to FP64 accuracy.  Each row r of P is written exactly as
//     P_r = 2^(e_r - 1021) sum_{s=1..7} q_rs 2^(-8 s),   q_rs integer, |q_rs| <= 128,
// from the bits of its FP64 values aligned to the row's largest biased exponent e_r (rounded
// to nearest at 2^-55 of the row maximum): a 55-bit integer per value, cut into seven
// balanced base-256 digits (the lower six in [-128, 127], the top one in [0, 128]), each
// exact in bf16.  A slice product Q_s Q_t^T sums W = 32 products of at most 2^14, so every
// group G_g = sum_{s+t=g} Q_s Q_t^T with g <= 9 (at most 7 terms) is an integer below 2^22
// and accumulates exactly in FP32; groups g >= 10 are below 2^-64 relative and dropped.  The
// FP64 update is
//     C_rc -= 2^(e_r + e_c - 2042) sum_g 2^(-8 g) G_g,rc.
// The eight groups are joined into one 64-bit integer w (join_groups, where they are counted from 0),
// pairs of them in 32 bits first; the lower four are rounded, by less than 2^-57 of the scale
// 2^(e_r + e_c - 2042).  The trailing matrix is held in the fixed point of kFixBits (assembled so
// by fit_instance): w is
// shifted to it and subtracted as an integer, so an updated entry costs no FP64 operation,
// and each block's columns are stored as FP64 by the update that completes them (the first block's
// by the assembly).  The slice products run on the tensor cores
// (trailing_update_tc); within a block the diagonal block is factorised in 8x8 tiles in shared
// memory and the rows below it are solved one row tile per warp (block_rows, FP64 pipe), which
// also writes their slices.
// Nt row tiles, of which the first Ntr are factorised (Nt > Ntr: appended query rows, whose
// rows below are solved and whose diagonal entries are updated, but not factorised).
template <class Tc>
__device__ bool factor_emulated(const SolveCtx& c, const Shared& s, double* A, int Nt, int Ntr, int* s_fail, Tc& tc) {
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarps = blockDim.x >> 5;
    const int g = lane >> 2, t = lane & 3;
    unsigned char* E = emu_ws(c);
    double* sr = emu_scales(c);           // row scales of the rows below the block
    double* Tall = emu_tile_inverses(c);  // inverses of all diagonal tiles, for the solves
    long long* udiag = emu_query_diag(c);
    auto tile = [&](int ir, int jc) { return s.Dblk + (ir * (ir + 1) / 2 + jc) * 64; };
    auto update = [&](int ir, int jc, int k) {  // tile (ir, jc) -= tile (ir, k) tile (jc, k)^T
        double* C = tile(ir, jc);
        double c0 = C[te(g, t)], c1 = C[te(g, 7 - t)];
        sub_products(c0, c1, tile(ir, k), g, tile(jc, k), t, 7 - t);
        C[te(g, t)] = c0;
        C[te(g, 7 - t)] = c1;
    };
    // the block's off-diagonal tiles and inverses to the workspace (for the solves and the cluster's
    // other CTAs) or from it
    auto exchange = [&](int K0, bool out) {
        const int nb = min(kEB, Ntr - K0);
        for (int x = tid; x < nb * (nb + 1) / 2 * 32; x += blockDim.x) {
            const int p = x >> 5, ir = tri_row(p), jc = p - ir * (ir + 1) / 2;
            double2* const g2 = reinterpret_cast<double2*>(ir == jc ? Tall + 64 * (K0 + ir) : A + eix(K0 + ir, K0 + jc));
            double2* const s2 = reinterpret_cast<double2*>(ir == jc ? s.Tblk + 64 * ir : tile(ir, jc));
            if (out)
                g2[x & 31] = s2[x & 31];
            else
                s2[x & 31] = g2[x & 31];
        }
    };
    // The diagonal block: tiles (it, jt), K0 <= jt <= it < K0 + kEB, in shared memory (packed),
    // right-looking by 8 columns.  Warp 0 takes the diagonal tiles; its update of the next one
    // needs no barrier after it.  The other tiles go to warps of the other sub-partitions
    // (warp 4 shares warp 0's), so the chain of diagonal tiles has its FP64 pipe alone.
    auto diagonal_block = [&](int K0) {
        const int nb = min(kEB, Ntr - K0);
        for (int x = tid; x < nb * (nb + 1) / 2 * 32; x += blockDim.x) {
            const int p = x >> 5, ir = tri_row(p), jc = p - ir * (ir + 1) / 2;
            reinterpret_cast<double2*>(s.Dblk)[x] = reinterpret_cast<const double2*>(A + eix(K0 + ir, K0 + jc))[x & 31];
        }
        __syncthreads();
        for (int k = 0; k < nb; ++k) {
            const double* Ti = s.Tblk + 64 * k;
            if (warp == 0) {
                if (k > 0) update(k, k, k - 1);
                __syncwarp();
                if (!diag_tile_warp<true>(tile(k, k), s.Tblk + 64 * k, s.invd + 8 * (K0 + k), s.dtab) && lane == 0)
                    *s_fail = 1;
            } else if (k > 0 && (warp & 3) != 0) {
                // the tiles (ir, jc), k <= jc <= ir, but (k, k): at most 5, one for each of warps 1, 2, 3, 5, 6
                const int m = nb - k, p = warp - (warp >> 2);
                if (p < m * (m + 1) / 2) {
                    const int ir = tri_row(p);
                    update(k + ir, k + p - ir * (ir + 1) / 2, k - 1);
                }
            }
            __syncthreads();
            if (*s_fail || k + 1 == nb) break;
            if (warp >= 1 && warp < nb - k) {  // panel: tile (k + warp, k) Ti^T
                double* T = tile(k + warp, k);
                double c0, c1;
                times_inverse(c0, c1, T, g, Ti, t, 7 - t);
                __syncwarp();
                T[te(g, t)] = c0;
                T[te(g, 7 - t)] = c1;
            }
            __syncthreads();
        }
        exchange(K0, true);
    };
    // In a cluster of four or more the first CTA looks ahead: it updates the tile that holds the next
    // diagonal block first and factorises that while the others take the rest of the update (the
    // diagonal block's chain of 32 columns, about 31k clocks, is as long as their share of it).
    const bool ahead = tc.n() >= 4;
    bool ok = true;
    for (int K0 = 0; K0 < Ntr; K0 += kEB) {
        const int K1 = min(K0 + kEB, Ntr);
        if (tc.rank() == 0 && (K0 == 0 || !ahead)) diagonal_block(K0);
        if (tc.n() > 1) {
            if (group_sync(tc, *s_fail || !ok)) {  // a pivot or, known to all after another barrier, a wait
                if (group_sync(tc, !ok)) emu_fail(c, tc);
                return false;
            }
            if (tc.rank() > 0) exchange(K0, false);
            __syncthreads();
        } else if (*s_fail) {
            return false;
        }
        if (K1 >= Nt) break;
        // the rows below: one warp per row tile solves its four tiles against the diagonal
        // block and writes their slices (both column halves) and row scales
        for (int it = K1 + warp + nwarps * tc.rank(); it < Nt; it += nwarps * tc.n())
            block_rows(A, it, K0, s.Dblk, s.Tblk, reinterpret_cast<double*>(s.stage) + kEB * 64 * warp,
                       reinterpret_cast<uint32_t*>(E + (int64_t)((it - K1) / kColT) * kGroupBytes +
                                                   (it - K1) % kColT * kSliceBytes),
                       sr + 8 * (it - K1),
                       it >= Ntr ? udiag + 8 * (it - Ntr) : nullptr);
        // the slices are read by the copy engine (async proxy)
        asm volatile("fence.proxy.async;" ::: "memory");
        group_barrier(tc);
        if (tc.n() > 1) asm volatile("fence.proxy.async;" ::: "memory");
        const bool first = ahead && tc.rank() == 0;
        if (!first || K1 < Ntr)
            ok = trailing_update_tc(A, Nt, Ntr, K1, E, sr, s.stage, tc, first ? 0 : ahead ? tc.rank() - 1 : tc.rank(),
                                    first ? 1 : ahead ? tc.n() - 1 : tc.n(),
                                    first ? TilePart::kFirst : ahead ? TilePart::kRest : TilePart::kAll);
        if (!ahead) {
            // (alone, the update's own last barrier is enough; together, the next diagonal block needs
            // every CTA's tiles)
            if (tc.n() > 1 ? group_sync(tc, !ok) : !ok) return emu_fail(c, tc);
        } else if (first && K1 < Ntr) {
            __syncthreads();
            if (ok) diagonal_block(K1);
        }
    }
    return true;
}

// The emulated kernel's solve for the right-hand side s.z, by the group's first CTA; the others take
// the solution from its shared memory.
template <class Tc>
__device__ void solve_group(const SolveCtx& c, const Shared& s, const double* A, int Nt, double* out, Tc& tc) {
    if (tc.rank() == 0) chol_solve_inv(s.z, s.Dsol, A, Nt, out, emu_tile_inverses(c));
    if (tc.n() == 1) return;
    group_sync(tc, 0);
    if (tc.rank() > 0) {
        const uint32_t from = peer_word(out, 0);
        for (int j = threadIdx.x; j < 8 * Nt; j += blockDim.x)
            asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(out[j]) : "r"(from + 8 * j) : "memory");
    }
    __syncthreads();
}

// Assemble A, factorise, solve alpha.  Returns false if a pivot was not positive.
// Local coordinates of the query at position p (id qid) of instance I (defined below).
__device__ __forceinline__ void query_local(const SolveCtx& c, int I, int64_t p, int64_t qid, double xl[3],
                                            int* qi = nullptr);

// Latent variance by bordering (emulated kernel, nq > 0 queries of instance I from position q0):
// the matrix is padded to Nr = 32 ceil(N / 32) rows and the kernel vectors k_a of the queries are
// appended as rows Nr + a, with k(x*, x*) = 1 on the diagonal.  Factorising only the first Nr
// columns turns row Nr + a into v_a = L^-1 k_a and leaves the Schur complement, whose diagonal
// entry is 1 - |v_a|^2 = u_a (Eq. 2).  Each appended row's arithmetic involves only that row and
// the instance's own rows, so u_a does not depend on the other queries.
template <bool kProps, bool kEmu = false, class Tc = EmuTc<false>>
__device__ bool fit_instance(const SolveCtx& c, const Shared& s, int N, int64_t base, Tc* tc = nullptr, int nq = 0,
                             int64_t q0 = 0, int I = 0) {
    const int tid = threadIdx.x, nt = blockDim.x;
    const int lane = tid & 31, warp = tid >> 5, nwarps = nt >> 5;
    const int g = lane >> 2, t = lane & 3;
    __shared__ int s_fail;
    const int Np = nq > 0 ? (N + 31) & ~31 : (N + 7) & ~7, Nt = Np >> 3;  // the instance's rows (Nr)
    const int Ntq = Nt + (nq + 7) / 8;                                   // with the appended rows
    const bool lattice = c.b.Xi != nullptr;
    for (int e = tid; e < 3 * N; e += nt) {
        double v = c.b.Xl[3 * base + e];
        s.X[e] = v;
        s.Xf[e] = (float)v;
        // the point's own FP32 world coordinate, recovered exactly (the FP64 local value
        // differs from it by the centre up to a rounding far below half an FP32 ulp)
        if (kEmu && !lattice) s.Xw[e] = (float)(v + (c.b.centre ? c.b.centre[3 * (int64_t)I + e % 3] : 0.0));
    }
    if (lattice)
        for (int e = tid; e < N; e += nt) {
            const char4 q = c.b.Xi[base + e];
            s.xi[e] = ((int)q.x + 16) | (((int)q.y + 16) << 8) | (((int)q.z + 16) << 16);
        }
    if (nq > 0)  // local coordinates of the appended queries (NaN: not finite, row left zero)
        for (int a = tid; a < nq; a += nt) {
            const int64_t p = q0 + a;
            const int64_t qid = c.b.qidx ? c.b.qidx[p] : p;
            double xl[3];
            int qi = 0;
            query_local(c, I, p, qid, xl, &qi);
            const bool fin = isfinite(xl[0]) && isfinite(xl[1]) && isfinite(xl[2]);
            if (lattice) {  // the lattice code (its bits: a tiny float, never NaN); [1]: finite flag
                s.qw[3 * a] = __int_as_float(qi);
                s.qw[3 * a + 1] = fin ? 0.f : NAN;
            } else {
                for (int k = 0; k < 3; ++k)
                    s.qw[3 * a + k] = fin ? (float)(xl[k] + (c.b.centre ? c.b.centre[3 * (int64_t)I + k] : 0.0)) : NAN;
            }
        }
    if (tid == 0) s_fail = 0;
    __syncthreads();
    double* A = s.A;
    // A = K + sigma^2 I in 8x8 tiles (Sec. III-A kernel, Eq. 1 noise term); padding rows and
    // columns are the identity so the padded factor is block-diagonal.  The emulated kernel
    // writes the fixed point of kfix_ff2 (appended query rows: the query's kernel values, 1
    // on the diagonal, and only the diagonal tiles of the query-by-query block).
    if constexpr (kEmu) {
        // strips of 8 columns of the 32x32 blocks, one per warp at a time: a row per lane (its
        // point in registers), the columns' points broadcast, whole lines written.  The first
        // block's columns are stored as FP64 tiles, the rest in the fixed point.
        const int nbr = (Ntq + 3) >> 2, nbc = (Nt + 3) >> 2;
        const int sq = nbc * (nbc + 1) / 2;  // blocks of the matrix itself; then nbc per block of query rows
        const int n_strip = 4 * (sq + (nbr - nbc) * nbc);
        const long long diag1 = fix_of_double(1.0 + c.P.s2);  // s2: sigma_prop^2 for properties
        for (int st = warp + nwarps * tc->rank(); st < n_strip; st += nwarps * tc->n()) {
            const int p = st >> 2, c0 = 8 * (st & 3);
            const int bi = p < sq ? tri_row(p) : nbc + (p - sq) / nbc;
            const int bj = p < sq ? p - bi * (bi + 1) / 2 : (p - sq) % nbc;
            const int i = 32 * bi + lane, a = i - Np;  // a >= 0: appended query row
            const bool qrow = nq > 0 && a >= 0;
            const bool live = qrow ? a < nq && !isnan(s.qw[3 * a + 1]) : i < N;
            double* B = A + bix(bi, bj);
            float rw[3] = {0.f, 0.f, 0.f};
            int rx = 0;
            if (live && lattice) rx = qrow ? __float_as_int(s.qw[3 * a]) : s.xi[i];
            if (live && !lattice)
                for (int k = 0; k < 3; ++k) rw[k] = qrow ? s.qw[3 * a + k] : s.Xw[3 * i + k];
            long long v[8];
            const int j0 = 32 * bj + c0;
            // (every entry of the strip is computed, without a branch, and replaced where it is not
            // a kernel value, so that the eight run interleaved)
            if (lattice) {
#pragma unroll
                for (int e = 0; e < 8; ++e) v[e] = live && j0 + e < N ? fix_of_double(c.P.lat_tab[lat_m(s.xi[j0 + e], rx)]) : 0;
            } else if (c.P.precision == VGP_MIXED) {
                const F2 rw2[3] = {pair2(rw[0]), pair2(rw[1]), pair2(rw[2])};
#pragma unroll
                for (int e = 0; e < 8; e += 2)
                    kfix_ff2(rw2, s.Xw + 3 * (j0 + e), pair2(c.P.inv2l2_hi), pair2(c.P.inv2l2_lo), s.Tff, v[e], v[e + 1]);
            } else if (qrow) {  // the query's FP64 local coordinates, formed as query_local forms them
                double xq[3];
                for (int k = 0; k < 3; ++k) xq[k] = (double)rw[k] - (c.b.centre ? c.b.centre[3 * (int64_t)I + k] : 0.0);
                for (int e = 0; e < 8; ++e) {
                    double r2 = 0.0;
                    for (int k = 0; k < 3; ++k) {
                        const double d = s.X[3 * (j0 + e) + k] - xq[k];
                        r2 += d * d;
                    }
                    v[e] = fix_of_double(exp(-r2 * c.P.inv2l2));
                }
            } else {
                for (int e = 0; e < 8; ++e) v[e] = j0 + e < i ? fix_of_double(exp(kval_arg(c.P, s, i, j0 + e))) : 0;
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) {
                const int j = j0 + e;
                if (!live || j >= N || (!qrow && j >= i)) v[e] = qrow || i != j ? 0 : i < N ? diag1 : 1ll << kFixBits;
            }
            if (bj == 0) {
                double* T = B + (c0 >> 3) * kTileCol + (lane >> 3) * 64;
#pragma unroll
                for (int e = 0; e < 8; e += 2)
                    *reinterpret_cast<double2*>(T + te(lane & 7, e)) = make_double2(double_of_fix(v[e]), double_of_fix(v[e + 1]));
            } else {
                long long* F = reinterpret_cast<long long*>(B) + 32 * c0 + lane;
#pragma unroll
                for (int e = 0; e < 8; ++e) F[32 * e] = v[e];
            }
        }
        if (nq > 0)
            for (int a = tid; a < 8 * (Ntq - Nt) && tc->rank() == 0; a += nt) emu_query_diag(c)[a] = 1ll << kFixBits;
        group_barrier(*tc);
    }
    if constexpr (!kEmu) {
        for (int64_t tl = warp; tl < n_tiles(Nt); tl += nwarps) {
            const int it = tri_row((int)tl), jt = (int)tl - it * (it + 1) / 2;
            for (int e = lane; e < 64; e += 32) {
                const int i = 8 * it + (e >> 3), j = 8 * jt + (e & 7);
                double v;
                if (i >= N || j >= N) v = (i == j) ? 1.0 : 0.0;
                else if (j > i) v = 0.0;
                else if (j == i) v = 1.0 + c.P.s2;
                else v = kval_pair(c.P, s, lattice, i, j);
                A[tl * 64 + te(e >> 3, e & 7)] = v;
            }
        }
    }
    __syncthreads();
    if (kEmu) {
        if (!factor_emulated(c, s, A, Ntq, Nt, &s_fail, *tc)) return false;
        // the staging of the tensor-core updates overwrote X, Xf and xi: reload them
        for (int e = tid; e < 3 * N; e += nt) {
            double v = c.b.Xl[3 * base + e];
            s.X[e] = v;
            s.Xf[e] = (float)v;
        }
        if (lattice)
            for (int e = tid; e < N; e += nt) {
                const char4 q = c.b.Xi[base + e];
                s.xi[e] = ((int)q.x + 16) | (((int)q.y + 16) << 8) | (((int)q.z + 16) << 16);
            }
        __syncthreads();
    } else
    for (int kt = 0; kt < Nt; ++kt) {
        // diagonal tile: 8x8 Cholesky and the inverse of its factor, by one warp, another one for each
        // tile and CTA so that the resident CTAs' tiles spread over the sub-partitions
        if (warp == (int)((kt + blockIdx.x) % nwarps)) {
            double* D = A + tix(kt, kt);
            if (s.Dsc) {
                reinterpret_cast<double2*>(s.Dsc)[lane] = reinterpret_cast<const double2*>(D)[lane];
                __syncwarp();
            }
            const bool good = diag_tile_warp<false>(s.Dsc ? s.Dsc : D, s.Tinv, s.invd + 8 * kt, s.dtab);
            if (s.Dsc) reinterpret_cast<double2*>(D)[lane] = reinterpret_cast<const double2*>(s.Dsc)[lane];
            if (!good && lane == 0) s_fail = 1;
        }
        __syncthreads();
        if (s_fail) break;
        // panel: L_it,kt = A_it,kt * Tinv^T (kept in shared memory too when A is global)
        for (int it = kt + 1 + warp; it < Nt; it += nwarps) {
            double* T = A + tix(it, kt);
            double c0, c1;
            times_inverse(c0, c1, T, g, s.Tinv, t, 7 - t);
            __syncwarp();
            T[te(g, t)] = c0;
            T[te(g, 7 - t)] = c1;
            if (s.panel) {
                double* Pt = s.panel + (it - kt - 1) * 64;
                Pt[te(g, t)] = c0;
                Pt[te(g, 7 - t)] = c1;
            }
        }
        __syncthreads();
        // trailing update A_it,jt -= L_it,kt L_jt,kt^T (kt < jt <= it) in 2x2 blocks of tiles per
        // warp, lane (g, t) row g and columns t, 7 - t of each: eight chains of fused multiply-adds
        // (the FP64 MMAs' own order and rounding; an 8x8x4 MMA takes 580 clocks for what eight of
        // these do in 528), six 16-byte operand loads for sixteen of them
        const int M = Nt - kt - 1;
        const int MB = (M + 1) >> 1;
        const int NB = MB * (MB + 1) / 2;
        for (int p = warp; p < NB; p += nwarps) {
            const int bi = tri_row(p), bj = p - bi * (bi + 1) / 2;
            const double *Pi[2], *Pj[2];
            double* C[2][2];
            bool valid[2][2];
            double acc[2][2][2];
#pragma unroll
            for (int r = 0; r < 2; ++r) {
                const int ii = min(2 * bi + r, M - 1), jj = min(2 * bj + r, M - 1);
                Pi[r] = s.panel ? s.panel + ii * 64 : A + tix(kt + 1 + ii, kt);
                Pj[r] = s.panel ? s.panel + jj * 64 : A + tix(kt + 1 + jj, kt);
            }
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int q = 0; q < 2; ++q) {
                    const int ii = 2 * bi + r, jj = 2 * bj + q;
                    valid[r][q] = ii < M && jj <= ii;
                    C[r][q] = A + (valid[r][q] ? tix(kt + 1 + ii, kt + 1 + jj) : tix(kt + 1 + 2 * bi, kt + 1 + 2 * bj));
                    acc[r][q][0] = C[r][q][te(g, t)];
                    acc[r][q][1] = C[r][q][te(g, 7 - t)];
                }
            // (a block on the diagonal has no upper right tile, the last row of blocks may have
            // no lower ones)
            const bool full = valid[0][1] && valid[1][0];
            if (full) {
#pragma unroll
                for (int m = 0; m < 8; m += 2) {
                    double2 x[2], u[2], v[2];
#pragma unroll
                    for (int r = 0; r < 2; ++r) {
                        x[r] = *reinterpret_cast<const double2*>(Pi[r] + te(g, m));
                        u[r] = *reinterpret_cast<const double2*>(Pj[r] + te(t, m));
                        v[r] = *reinterpret_cast<const double2*>(Pj[r] + te(7 - t, m));
                    }
#pragma unroll
                    for (int r = 0; r < 2; ++r)
#pragma unroll
                        for (int q = 0; q < 2; ++q) {
                            acc[r][q][0] = fma(-x[r].x, u[q].x, acc[r][q][0]);
                            acc[r][q][1] = fma(-x[r].x, v[q].x, acc[r][q][1]);
                        }
#pragma unroll
                    for (int r = 0; r < 2; ++r)
#pragma unroll
                        for (int q = 0; q < 2; ++q) {
                            acc[r][q][0] = fma(-x[r].y, u[q].y, acc[r][q][0]);
                            acc[r][q][1] = fma(-x[r].y, v[q].y, acc[r][q][1]);
                        }
                }
            } else {
#pragma unroll
                for (int r = 0; r < 2; ++r)
#pragma unroll
                    for (int q = 0; q < 2; ++q)
                        if (valid[r][q]) sub_products(acc[r][q][0], acc[r][q][1], Pi[r], g, Pj[q], t, 7 - t);
            }
#pragma unroll
            for (int r = 0; r < 2; ++r)
#pragma unroll
                for (int q = 0; q < 2; ++q)
                    if (valid[r][q]) {
                        C[r][q][te(g, t)] = acc[r][q][0];
                        C[r][q][te(g, 7 - t)] = acc[r][q][1];
                    }
        }
        __syncthreads();
    }
    if (s_fail) return false;
    // The solves use the instance's own 8-row tiles only: the leading block of the factor is the
    // factor of the leading block, so rows padded to 32 for appended queries change no bit of
    // alpha (the solves' work split depends on the tile count).
    const int Ns = (N + 7) & ~7, Nts = Ns >> 3;
    if (kProps) {
        // property weights alpha_c = A^-1 y_c, one right-hand side per channel (Eq. 6)
        for (int ch = 0; ch < c.b.nprop; ++ch) {
            for (int i = tid; i < Ns; i += nt) s.z[i] = i < N ? c.b.yprop[(base + i) * c.b.nprop + ch] : 0.0;
            __syncthreads();
            if constexpr (kEmu)
                solve_group(c, s, A, Nts, s.pa[ch], *tc);
            else
                chol_solve(s, A, Nts, s.pa[ch]);
        }
        return true;
    }
    // alpha = A^-1 1 (Eq. 1)
    for (int i = tid; i < Ns; i += nt) s.z[i] = i < N ? 1.0 : 0.0;
    __syncthreads();
    if constexpr (kEmu)
        solve_group(c, s, A, Nts, s.alpha, *tc);
    else
        chol_solve(s, A, Nts, s.alpha);
    for (int j = tid; j < Ns; j += nt) {
        const float hi = (float)s.alpha[j];
        s.alf[j] = hi;
        s.alf_lo[j] = (float)(s.alpha[j] - (double)hi);
    }
    __syncthreads();
    return true;
}

// Queries of a work item on an instance of N points (see k_chunk_plan).
__host__ __device__ __forceinline__ long long chunk_len(long long qc, int qn, long long N, int cap) {
    const long long q = qc > qn * N ? qc : qn * N;
    return cap > 0 && q > cap ? cap : q;
}

// The shortest work item worth a fit, chunk_len(qmin, qn, N, cap) queries, in the plain kernel or the
// emulated one:
// * Emulated launches with variance or properties: an appended row of an N-point instance costs about
//   1 / N of its fit; at least 64 of them, and at most what a factorisation appends.
// * Plain launches with variance run on the FP64 pipe; 128 queries.
// * The mean alone costs about N FP32 values a query: a fit is worth about 64 N of them.
struct ChunkRule {
    int qmin, qn, cap;
};
__host__ __device__ __forceinline__ ChunkRule chunk_rule(bool heavy, bool var, bool emu) {
    return {heavy && !emu ? 128 : 64, !heavy ? 64 : emu ? 1 : 0, emu && var ? kBorderQ : 0};
}

struct EvalOut {
    double d, g[3], v;
    int status;
};

// Reverting (Eq. 3), distance variance (Eq. 4), chain-rule gradient, with the caps of the
// occupancy: lo = log o, gro = grad o / o.
__device__ __forceinline__ void revert(const DevParams& P, double lo, const double gro[3], double u, bool want_var,
                                       EvalOut& r) {
    if (!(lo >= P.log_floor)) {  // also catches NaN (o <= 0)
        r.status = VGP_ST_CLAMPED;
        r.d = P.d_max;
        r.g[0] = r.g[1] = r.g[2] = 0.0;
        r.v = INFINITY;
        return;
    }
    r.status = VGP_ST_OK;
    if (lo >= 0.0) {
        const double lam = -P.l2 / P.d_var_floor;
        r.d = 0.0;
        r.g[0] = r.g[1] = r.g[2] = 0.0;
        r.v = want_var ? lam * lam * u : NAN;
        return;
    }
    const double d = sqrt(-2.0 * P.l2 * lo);
    r.d = d;
    for (int a = 0; a < 3; ++a) r.g[a] = -P.l2 * gro[a] / d;
    if (want_var) {
        const double o = exp(lo);
        const double lam = -P.l2 / (o * fmax(d, P.d_var_floor));
        r.v = lam * lam * u;
    } else {
        r.v = NAN;
    }
}

__device__ __forceinline__ void write_out(const SolveBatch& b, int64_t qid, const EvalOut& r) {
    b.d[qid] = r.d;
    if (b.grad) {
        b.grad[3 * qid] = r.g[0];
        b.grad[3 * qid + 1] = r.g[1];
        b.grad[3 * qid + 2] = r.g[2];
    }
    if (b.var) b.var[qid] = r.v;
    if (b.status) b.status[qid] = (uint8_t)r.status;
}

__device__ __forceinline__ void query_local(const SolveCtx& c, int I, int64_t p, int64_t qid, double xl[3],
                                            int* qi) {
    double xg[3];
    if (c.b.qkey) {
        int i, j, k;
        unpack_key(c.b.qkey[p], i, j, k);
        if (qi && c.b.inst_key) {
            int lx, ly, lz;
            unpack_key(c.b.inst_key[I], lx, ly, lz);
            // offsets relative to the instance leaf origin, biased by 16 into 0..255
            *qi = (i - 8 * lx + 16) | ((j - 8 * ly + 16) << 8) | ((k - 8 * lz + 16) << 16);
        }
        xg[0] = (double)i * c.P.vs;
        xg[1] = (double)j * c.P.vs;
        xg[2] = (double)k * c.P.vs;
    } else {
        const int64_t qp = qid / c.b.qdiv;
        xg[0] = (double)c.b.qxyz[3 * qp];
        xg[1] = (double)c.b.qxyz[3 * qp + 1];
        xg[2] = (double)c.b.qxyz[3 * qp + 2];
    }
    for (int a = 0; a < 3; ++a) xl[a] = xg[a] - c.b.centre[3 * (int64_t)I + a];
}

// Mixed precision: latent mean and gradient at one query as sums of kernel values scaled by
// e^(r0^2 / 2l^2): tot = o times that (FP64 sum of two floats), g = l^2 grad o times it.
// qi: biased lattice offsets of the query (lattice instances only; r0 = 0 there).
// FP32 kernel values and FP32 accumulation.  Off the lattice, the nearest training point shifts the
// exponent (exp(-(r^2 - r0^2) / 2l^2) <= 1, no underflow).  The sum is compensated: alpha is carried
// as two floats and the rounding error of every product and addition is accumulated separately
// (Neumaier), all on the FP32 pipe.
__device__ __forceinline__ void mean_mixed(const DevParams& P, const Shared& s, int N, bool lattice, int qi,
                                           const double xl[3], float& r0, double& tot, float g[3]) {
    const float qx = (float)xl[0], qy = (float)xl[1], qz = (float)xl[2];
    r0 = 0.f;
    if (!lattice) {
        r0 = INFINITY;
        for (int j = 0; j < N; ++j) {
            float dx = s.Xf[3 * j] - qx, dy = s.Xf[3 * j + 1] - qy, dz = s.Xf[3 * j + 2] - qz;
            r0 = fminf(r0, fmaf(dx, dx, fmaf(dy, dy, dz * dz)));
        }
    }
    float sum = 0.f, comp = 0.f, gx = 0.f, gy = 0.f, gz = 0.f;
    for (int j = 0; j < N; ++j) {
        float dx = s.Xf[3 * j] - qx, dy = s.Xf[3 * j + 1] - qy, dz = s.Xf[3 * j + 2] - qz;
        float e;
        if (lattice) {
            e = P.lat_tab_f[lat_m(s.xi[j], qi)];
        } else {
            float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
            e = exp2f((r0 - r2) * P.inv2l2_log2e);
        }
        const float ah = s.alf[j];
        const float w = ah * e;
        comp += fmaf(ah, e, -w) + s.alf_lo[j] * e;
        const float t2 = sum + w;
        comp += fabsf(sum) >= fabsf(w) ? (sum - t2) + w : (w - t2) + sum;
        sum = t2;
        gx = fmaf(w, dx, gx);
        gy = fmaf(w, dy, gy);
        gz = fmaf(w, dz, gz);
    }
    tot = (double)sum + (double)comp;
    g[0] = gx;
    g[1] = gy;
    g[2] = gz;
}

// revert() of mean_mixed's sums without the variance: o = tot e^(-r0^2 / 2l^2), grad d = -l^2 grad o /
// (o d) = -g / (tot d), d exactly as revert() forms it.  An FP64 operation is worth 66 FP32
// instructions here: one division serves the three components instead of four (about 60 operations a
// query with the logarithm instead of 95; 4M evaluations of 61 points: 1.49 -> 1.1 ms).
__device__ __forceinline__ void revert_mixed(const DevParams& P, float r0, double tot, const float g[3], EvalOut& r) {
    const double lo = tot > 0.0 ? -(double)r0 * P.inv2l2 + log(tot) : NAN;
    if (!(lo >= P.log_floor) || lo >= 0.0) {
        const double none[3] = {0.0, 0.0, 0.0};
        revert(P, lo, none, 0.0, false, r);
        return;
    }
    const double d = sqrt(-2.0 * P.l2 * lo), w = -1.0 / (tot * d);
    r.status = VGP_ST_OK;
    r.d = d;
    for (int a = 0; a < 3; ++a) r.g[a] = w * (double)g[a];
    r.v = NAN;
}

// FP64 latent mean and gradient at one query; returns lo = log o and gro = grad o / o.
__device__ __forceinline__ void latent_mean(const DevParams& P, const Shared& s, int N, bool lattice, int qi,
                                            const double xl[3], double& lo, double gro[3]) {
    double o = 0.0, gx = 0.0, gy = 0.0, gz = 0.0;
    for (int j = 0; j < N; ++j) {
        double dx = s.X[3 * j] - xl[0], dy = s.X[3 * j + 1] - xl[1], dz = s.X[3 * j + 2] - xl[2];
        double k;
        if (lattice) k = P.lat_tab[lat_m(s.xi[j], qi)];
        else k = exp(-(dx * dx + dy * dy + dz * dz) * P.inv2l2);
        const double w = s.alpha[j] * k;
        o += w;
        gx += w * dx;
        gy += w * dy;
        gz += w * dz;
    }
    if (!(o > 0.0)) {
        lo = NAN;
        gro[0] = gro[1] = gro[2] = 0.0;
        return;
    }
    lo = log(o);
    const double inv = 1.0 / (o * P.l2);
    gro[0] = gx * inv;
    gro[1] = gy * inv;
    gro[2] = gz * inv;
}

// u = 1 - |L^-1 k|^2 (Eq. 2) with FP64 kernel values; the thread's own column of V lives in
// global workspace.
__device__ __forceinline__ double latent_var(const DevParams& P, const Shared& s, int N, bool lattice, int qi,
                                             const double xl[3], double* V, int stride) {
    const double* A = s.A;
    double acc = 0.0;
    for (int i = 0; i < N; ++i) {
        double sum;
        if (lattice) {
            sum = P.lat_tab[lat_m(s.xi[i], qi)];
        } else {
            double dx = s.X[3 * i] - xl[0], dy = s.X[3 * i + 1] - xl[1], dz = s.X[3 * i + 2] - xl[2];
            const double y = -(dx * dx + dy * dy + dz * dz) * P.inv2l2;
            sum = P.precision == VGP_MIXED ? exp_neg(y, s.T256) : exp(y);
        }
        const int it = i >> 3, r = i & 7;
        for (int jt = 0; jt < it; ++jt) {
            const double* T = A + tix(it, jt);
#pragma unroll
            for (int c2 = 0; c2 < 8; ++c2) sum -= T[te(r, c2)] * V[(int64_t)(8 * jt + c2) * stride];
        }
        const double* T = A + tix(it, it);
        for (int c2 = 0; c2 < r; ++c2) sum -= T[te(r, c2)] * V[(int64_t)(8 * it + c2) * stride];
        const double vi = sum * s.invd[i];
        V[(int64_t)i * stride] = vi;
        acc += vi * vi;
    }
    return fmax(0.0, 1.0 - acc);
}

// Property means c_ch = sum_j alpha_ch,j k_j (Eq. 6) in FP64 with FP64 kernel values.
__device__ __forceinline__ void property_mean(const DevParams& P, const Shared& s, int N, int nprop,
                                              bool lattice, int qi, const double xl[3], double* out) {
    double acc[4] = {0.0, 0.0, 0.0, 0.0};
    for (int j = 0; j < N; ++j) {
        double k;
        if (lattice) {
            k = P.lat_tab[lat_m(s.xi[j], qi)];
        } else {
            double dx = s.X[3 * j] - xl[0], dy = s.X[3 * j + 1] - xl[1], dz = s.X[3 * j + 2] - xl[2];
            k = exp(-(dx * dx + dy * dy + dz * dz) * P.inv2l2);
        }
#pragma unroll
        for (int ch = 0; ch < 4; ++ch)
            if (ch < nprop) acc[ch] += s.pa[ch][j] * k;
    }
#pragma unroll
    for (int ch = 0; ch < 4; ++ch)
        if (ch < nprop) out[ch] = acc[ch];
}

__device__ __forceinline__ void invalid(EvalOut& r, int status) {
    r.status = status;
    r.d = INFINITY;
    r.g[0] = r.g[1] = r.g[2] = 0.0;
    r.v = INFINITY;
}

// The body of the GP solve kernels (see k_solve below).
template <bool kProps, bool kEmu, bool kGroup>
__device__ __forceinline__ void solve_body(const SolveCtx& c) {
    extern __shared__ __align__(128) double sm[];
    __shared__ int s_item[2];
    __shared__ uint32_t s_tmem;
    __shared__ __align__(8) uint64_t s_bar[2];
    const int tid = threadIdx.x, nt = blockDim.x;
    __shared__ int s_flags[2 * 8];
    const int ncta = kGroup ? c.ncta : 1;
    const int group = (int)blockIdx.x / ncta, n_groups = (int)gridDim.x / ncta;  // CTAs that share work items
    double* ws_a = c.a_in_smem ? nullptr : c.ws_a + (int64_t)group * c.ws_a_stride;
    Shared s = carve(sm, c.npad, c.a_in_smem, ws_a, c.b.nprop, c.stage_panel, c.b.Xi != nullptr, false, kEmu);
    double* V = c.ws_v ? c.ws_v + (int64_t)blockIdx.x * c.ws_v_stride + tid : nullptr;
    const bool lattice = c.b.Xi != nullptr;
    for (int j = tid; j < 256; j += nt) {
        if constexpr (kEmu) {
            float h, l;
            split_pair(c.P.exp_tab[j], h, l);
            s.Tff[j] = make_float2(h, l);
        } else {
            s.T256[j] = c.P.exp_tab[j];
        }
    }
    for (int j = tid; j < 256; j += nt) s.dtab[j] = diag_entry(j >> 5, j & 31);
    EmuTc<kGroup> tc{};
    tc.n_ = ncta;
    tc.rank_ = (int)blockIdx.x % ncta;
    tc.flags = s_flags;
    if (kEmu) {
        // tensor memory for the 8 slice-group accumulators (held until the CTA exits) and the
        // barriers of the staging copies and of the MMAs
        if ((tid >> 5) == 0) {
            asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&s_tmem)),
                         "r"(kEmuTmemCols)
                         : "memory");
            asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
        }
        if (tid == 0) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&s_bar[0])) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&s_bar[1])) : "memory");
            asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        }
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        tc.tmem = s_tmem;
        tc.bar_ld = smem_addr(&s_bar[0]);
        tc.bar_mma = smem_addr(&s_bar[1]);
        if (tc.n() > 1) {  // every CTA of the cluster runs before another one writes to its shared memory
            asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory");
            asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
        }
    }
    for (bool first = true;; first = false) {
        // the next work item: an instance, or one chunk of its queries (the instance is fitted
        // again for every chunk, so the queries of a large instance spread over the GPU).  CTA i
        // takes item i first (the CTAs of a launch are spread over the SMs in index order, so a
        // grid larger than the work stays balanced), then items from the counter.
        if (tid == 0 && tc.rank() == 0) {
            const int w = first ? group : n_groups + atomicAdd(c.counter, 1);
            // graph mode: this bucket's count and share of the order, planned on the device
            const int nb = c.plan ? c.plan[c.bucket] : c.n_work;
            const int ob = c.plan ? c.plan[5 + c.bucket] : 0;
            int k = w, ci = 0, nw = nb;
            if (c.chunk_off) {
                const int* cof = c.chunk_off + ob;  // direct launches pass the bucket's offset
                nw = cof[nb] - cof[0];
                if (w < nw) {  // the last instance whose first chunk is at or before w
                    const int t = cof[0] + w;
                    int lo = 0, hi = nb - 1;
                    while (lo < hi) {
                        const int mid = (lo + hi + 1) >> 1;
                        if (cof[mid] <= t)
                            lo = mid;
                        else
                            hi = mid - 1;
                    }
                    k = lo;
                    ci = t - cof[lo];
                }
            }
            s_item[0] = w < nw ? (c.order ? c.order[ob + k] : c.inst_base + k) : -1;
            s_item[1] = ci;
            if constexpr (kEmu)
                for (int r = 1; r < tc.n(); ++r) {
                    peer_store(&s_item[0], r, s_item[0]);
                    peer_store(&s_item[1], r, s_item[1]);
                }
        }
        if constexpr (kEmu)
            group_barrier(tc);
        else
            __syncthreads();
        const int I = s_item[0], ci = s_item[1];
        if constexpr (kEmu)
            group_barrier(tc);
        else
            __syncthreads();
        if (I < 0) break;
        const int64_t base = c.b.inst_off[I];
        const int N = (int)(c.b.inst_off[I + 1] - base);
        const int64_t qa = c.b.q_off[I], qb = c.b.q_off[I + 1];
        const int qc = c.chunk_q ? *c.chunk_q : 0;
        const int64_t qch = qc > 0 ? chunk_len(qc, c.chunk_qn, N, c.chunk_cap) : 0;
        const int64_t q0 = qch > 0 ? min(qb, qa + ci * qch) : qa;
        const int64_t q1 = qch > 0 ? min(qb, q0 + qch) : qb;
        if (kProps) {
            // property mode: means and variance (Eq. 6, variance read as for Eq. 2).  The emulated
            // kernel takes the variance by bordering, chunk by chunk (see below), on the property
            // GP's own matrix (noise sigma_c^2)
            const int np = c.b.nprop;
            for (int64_t cq0 = q0;;) {
                const int64_t cq1 = kEmu ? min(q1, cq0 + (int64_t)c.qmax) : q1;
                const bool ok = N > 0 && fit_instance<kProps, kEmu>(c, s, N, base, &tc, kEmu ? (int)(cq1 - cq0) : 0, cq0, I);
                const int64_t ce = ok ? cq1 : q1;  // a failed factorisation answers all remaining queries
                for (int64_t p = cq0 + tid + (int64_t)nt * tc.rank(); p < ce; p += nt * tc.n()) {
                    const int64_t qid = c.b.qidx ? c.b.qidx[p] : p;
                    double xl[3], cm[4] = {NAN, NAN, NAN, NAN}, w = INFINITY;
                    int qi = 0;
                    if (ok) {
                        query_local(c, I, p, qid, xl, &qi);
                        if (isfinite(xl[0]) && isfinite(xl[1]) && isfinite(xl[2])) {
                            property_mean(c.P, s, N, np, lattice, qi, xl, cm);
                            if constexpr (kEmu)
                                w = fmax(0.0, double_of_fix(emu_query_diag(c)[p - cq0]));
                            else
                                w = latent_var(c.P, s, N, lattice, qi, xl, V, nt);
                        }
                    }
                    for (int ch = 0; ch < np; ++ch) c.b.pc[qid * np + ch] = cm[ch];
                    c.b.pw[qid] = w;
                }
                if (!ok && N > 0 && tid == 0 && !tc.dead) atomicOr(c.err, kErrFactor);
                if constexpr (kEmu)
                    group_barrier(tc);
                else
                    __syncthreads();
                cq0 = ce;
                if ((kEmu && tc.dead) || cq0 >= q1) break;
            }
            if (kEmu && tc.dead) break;
            continue;
        }
        // Variance by bordering (see fit_instance): the instance's queries are appended to its
        // matrix in chunks of at most qmax, one factorisation per chunk.  Every chunk repeats
        // the same arithmetic on the instance's own rows, and a query's row involves only
        // itself, so every result is independent of the chunking and of the other queries.
        const bool border = kEmu && c.b.want_var;
        for (int64_t cq0 = q0;;) {
            const int64_t cq1 = border ? min(q1, cq0 + (int64_t)c.qmax) : q1;
            const bool ok = N > 0 && fit_instance<kProps, kEmu>(c, s, N, base, &tc, border ? (int)(cq1 - cq0) : 0,
                                                                 cq0, I);
            if (c.b.alpha_out && ci == 0 && cq0 == q0 && tc.rank() == 0)
                for (int j = tid; j < N; j += nt) c.b.alpha_out[base + j] = ok ? s.alpha[j] : NAN;
            const int64_t ce = ok ? cq1 : q1;  // a failed factorisation answers all remaining queries
            for (int64_t p = cq0 + tid + (int64_t)nt * tc.rank(); p < ce; p += nt * tc.n()) {
                const int64_t qid = c.b.qidx ? c.b.qidx[p] : p;
                EvalOut r;
                if (!ok) {
                    invalid(r, N > 0 ? VGP_ST_FACTOR_FAIL : VGP_ST_NO_SUPPORT);
                } else {
                    double xl[3], lo, gro[3];
                    int qi = 0;
                    query_local(c, I, p, qid, xl, &qi);
                    if (!(isfinite(xl[0]) && isfinite(xl[1]) && isfinite(xl[2]))) {
                        invalid(r, VGP_ST_BAD_INPUT);
                    } else {
                        double u = 0.0;
                        if (c.b.want_var) {
                            if constexpr (kEmu)  // the Schur complement's diagonal entry, clamped at 0
                                u = fmax(0.0, double_of_fix(emu_query_diag(c)[p - cq0]));
                            else
                                u = latent_var(c.P, s, N, lattice, qi, xl, V, nt);
                        }
                        if (c.P.precision == VGP_MIXED) {
                            float r0, g[3];
                            double tot;
                            mean_mixed(c.P, s, N, lattice, qi, xl, r0, tot, g);
                            if (!c.b.want_var) {
                                revert_mixed(c.P, r0, tot, g, r);
                            } else {
                                lo = tot > 0.0 ? -(double)r0 * c.P.inv2l2 + log(tot) : NAN;
                                const double inv = 1.0 / (tot * c.P.l2);
                                for (int a = 0; a < 3; ++a) gro[a] = (double)g[a] * inv;
                                revert(c.P, lo, gro, u, true, r);
                            }
                        } else {
                            latent_mean(c.P, s, N, lattice, qi, xl, lo, gro);
                            revert(c.P, lo, gro, u, c.b.want_var != 0, r);
                        }
                    }
                }
                write_out(c.b, qid, r);
            }
            if (!ok && N > 0 && tid == 0 && !tc.dead) atomicOr(c.err, kErrFactor);
            if constexpr (kEmu)
                group_barrier(tc);
            else
                __syncthreads();
            cq0 = ce;
            if ((kEmu && tc.dead) || cq0 >= q1) break;
        }
        if (kEmu && tc.dead) break;
    }
    if (kEmu) {
        if (tc.dead) {  // let copies or MMAs still in flight finish (bounded) before releasing
            bar_wait(tc.bar_ld, tc.ph_ld);
            bar_wait(tc.bar_mma, tc.ph_mma);
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncthreads();
        if ((tid >> 5) == 0)
            asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tc.tmem), "r"(kEmuTmemCols)
                         : "memory");
    }
}

// kProps: surface-property mode (Eq. 6); the emulated kernels run the trailing updates of
// N > 32 instances on the bf16 tensor cores (256 threads, two CTAs per SM).  Separate
// kernels, so that the plain distance kernel keeps its register budget.
template <bool kProps>
__global__ void __launch_bounds__(kPlainThreads) k_solve(SolveCtx c) {
    solve_body<kProps, false, false>(c);
}

template <bool kProps, bool kGroup>
__global__ void __launch_bounds__(kEmuThreads, 2) k_solve_emu(SolveCtx c) {
    solve_body<kProps, true, kGroup>(c);
}

// Backward pass (derived from Eq. 1 and Eq. 3): per instance,
//   obar_q = dL/dd_q * dd/do_q, abar = sum_q obar_q k_q, lambda = A^-1 abar,
//   dL/dx_j = sum_q obar_q alpha_j k_qj (x*_q - x_j) / l^2
//             - sum_i (lambda_i alpha_j + lambda_j alpha_i) k_ij (x_i - x_j) / l^2,
// and dL/dx*_q = dL/dd_q grad d_q.  FP64 throughout; alpha is recomputed, not stored.
__global__ void k_backward(SolveCtx c) {
    extern __shared__ double sm[];
    __shared__ int s_w;
    const int tid = threadIdx.x, nt = blockDim.x;
    double* ws_a = c.a_in_smem ? nullptr : c.ws_a + (int64_t)blockIdx.x * c.ws_a_stride;
    Shared s = carve(sm, c.npad, c.a_in_smem, ws_a, 0, c.stage_panel, c.b.Xi != nullptr, true);
    const double l2 = c.P.l2;
    SolveCtx cc = c;
    cc.P.precision = VGP_FP64;
    for (int j = tid; j < 256; j += nt) {
        s.T256[j] = c.P.exp_tab[j];
        s.dtab[j] = diag_entry(j >> 5, j & 31);
    }
    __syncthreads();
    for (;;) {
        if (tid == 0) s_w = atomicAdd(c.counter, 1);
        __syncthreads();
        const int w = s_w;
        __syncthreads();
        if (w >= c.n_work) break;
        const int I = c.order[w];
        const int64_t base = c.b.inst_off[I];
        const int N = (int)(c.b.inst_off[I + 1] - base);
        const int Nt = (N + 7) >> 3;
        const int64_t q0 = c.b.q_off[I], q1 = c.b.q_off[I + 1];
        const bool ok = N > 0 && fit_instance<false>(cc, s, N, base);
        for (int64_t p = q0 + tid; p < q1; p += nt) {
            const int64_t qid = c.b.qidx ? c.b.qidx[p] : p;
            double ob = 0.0, gq[3] = {0.0, 0.0, 0.0};
            if (ok) {
                double xl[3], lo, gro[3];
                query_local(cc, I, p, qid, xl);
                latent_mean(cc.P, s, N, false, 0, xl, lo, gro);
                EvalOut r;
                revert(cc.P, lo, gro, 0.0, false, r);
                const double gd = c.bw.dL_dd[qid];
                for (int a = 0; a < 3; ++a) gq[a] = gd * r.g[a];
                if (r.status == VGP_ST_OK && r.d > 0.0 && lo < 0.0) ob = gd * (-l2 / (exp(lo) * r.d));
            }
            c.bw.obar[p] = ob;
            if (c.bw.dL_dq)
                for (int a = 0; a < 3; ++a) c.bw.dL_dq[3 * qid + a] = gq[a];
        }
        __syncthreads();
        if (ok && c.bw.dL_dX) {
            // abar_j and the direct term, thread per training point
            for (int j = tid; j < 8 * Nt; j += nt) {
                if (j >= N) {
                    s.z[j] = 0.0;
                    continue;
                }
                double ab = 0.0, g1[3] = {0.0, 0.0, 0.0};
                for (int64_t p = q0; p < q1; ++p) {
                    const double ob = c.bw.obar[p];
                    if (ob == 0.0) continue;
                    const int64_t qid = c.b.qidx ? c.b.qidx[p] : p;
                    double xl[3];
                    query_local(cc, I, p, qid, xl);
                    double dx = xl[0] - s.X[3 * j], dy = xl[1] - s.X[3 * j + 1], dz = xl[2] - s.X[3 * j + 2];
                    double k = exp_near(-(dx * dx + dy * dy + dz * dz) * c.P.inv2l2, s.T256, c.P.exp_lo);
                    ab += ob * k;
                    g1[0] += ob * k * dx;
                    g1[1] += ob * k * dy;
                    g1[2] += ob * k * dz;
                }
                s.z[j] = ab;
                for (int a = 0; a < 3; ++a) g1[a] *= s.alpha[j] / l2;
                const int64_t gi = c.bw.gidx[base + j];
                for (int a = 0; a < 3; ++a) atomicAdd(&c.bw.dL_dX[3 * gi + a], g1[a]);
            }
            __syncthreads();
            chol_solve(s, s.A, Nt, s.w);  // lambda = A^-1 abar -> s.w
            for (int j = tid; j < N; j += nt) {
                double g2[3] = {0.0, 0.0, 0.0};
                const double lj = s.w[j], aj = s.alpha[j];
                for (int i = 0; i < N; ++i) {
                    if (i == j) continue;
                    double dx = s.X[3 * i] - s.X[3 * j], dy = s.X[3 * i + 1] - s.X[3 * j + 1],
                           dz = s.X[3 * i + 2] - s.X[3 * j + 2];
                    double k = exp_near(-(dx * dx + dy * dy + dz * dz) * c.P.inv2l2, s.T256, c.P.exp_lo);
                    double cf = (s.w[i] * aj + lj * s.alpha[i]) * k;
                    g2[0] -= cf * dx;
                    g2[1] -= cf * dy;
                    g2[2] -= cf * dz;
                }
                const int64_t gi = c.bw.gidx[base + j];
                for (int a = 0; a < 3; ++a) atomicAdd(&c.bw.dL_dX[3 * gi + a], g2[a] / l2);
            }
        }
        __syncthreads();
    }
}

// Instances of each size.  With more (1025 words, then five of 64 bits, 8-byte aligned): the work items
// beyond one per instance of each size, were every chunk the shortest (chunk_rule), and the
// queries of each size bucket (N > 224, > 128, > 64, > 32, the rest).
constexpr int kHistWords = 1026;  // (a word of padding)
__global__ void k_hist_n(const int64_t* inst_off, const int64_t* q_off, int64_t n, int* hist, int* more, bool heavy,
                         bool var, bool emulate) {
    __shared__ unsigned long long sum[5];
    if (threadIdx.x < 5) sum[threadIdx.x] = 0;
    __syncthreads();
    const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i < n) {
        const int N = (int)(inst_off[i + 1] - inst_off[i]);
        atomicAdd(&hist[min(N, 1024)], 1);
        if (more) {
            const int64_t nq = q_off[i + 1] - q_off[i];
            const int bk = N > 224 ? 0 : N > 128 ? 1 : N > 64 ? 2 : N > 32 ? 3 : 4;
            atomicAdd(&sum[bk], (unsigned long long)nq);
            const ChunkRule r = chunk_rule(heavy, var, emulate && N > 32);
            const long long len = chunk_len(r.qmin, r.qn, N, r.cap);
            if (nq > len) atomicAdd(&more[min(N, 1024)], (int)((nq - 1) / len));
        }
    }
    __syncthreads();
    if (more && threadIdx.x < 5 && sum[threadIdx.x])
        atomicAdd(reinterpret_cast<unsigned long long*>(more + kHistWords) + threadIdx.x, sum[threadIdx.x]);
}

// order[] sorted by increasing N via the prefix of the histogram
__global__ void k_order_n(const int64_t* inst_off, int64_t n, int* cursor, int32_t* order) {
    int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
    if (i >= n) return;
    int N = (int)(inst_off[i + 1] - inst_off[i]);
    int pos = atomicAdd(&cursor[min(N, 1024)], 1);
    order[pos] = (int32_t)i;
}

__global__ void k_or_err(int* err, int bits) { atomicOr(err, bits); }

// Device bucket plan (graph mode): cursor[N] = first position of size N in decreasing-N
// order; plan[b] = instances of bucket b, plan[5 + b] = its first position.
__global__ void k_plan_buckets(const int* hist, int* cursor, int* plan) {
    if (threadIdx.x != 0 || blockIdx.x != 0) return;
    int run = 0;
    for (int N = 1024; N >= 0; --N) {
        cursor[N] = run;
        run += hist[N];
    }
    const int lo[5] = {225, 129, 65, 33, 0}, hi[5] = {1024, 224, 128, 64, 32};
    int off = 0;
    for (int b = 0; b < 5; ++b) {
        int cnt = 0;
        for (int N = lo[b]; N <= hi[b]; ++N) cnt += hist[N];
        plan[b] = cnt;
        plan[5 + b] = off;
        off += cnt;
    }
}

// Work items of the solve launches: an instance's queries are split into chunks, so that they spread
// over the GPU; each chunk fits the instance again.  The chunk size of an instance of N points in
// launch b is max(qc, qn[b] N), qn N queries being what an evaluation has to be worth a fit
// (chunk_len).  qc is the smallest, from qmin[b], that gives no more chunks than the slots[b] CTAs
// that run at once, or slots[b] more than instances where those are more: the refits then run on CTAs
// that had no work, and the longest chunk, the launch's tail, is as short as can be.  cap[b] > 0
// bounds qc (the rows a bordered factorisation appends).  chunk_q[b] receives qc (0: no split);
// chunk_off[k] the number of work items of the order before instance k, chunk_off[n] the total.
// The buckets are contiguous in the order: from the device plan in graph mode, else from a.
struct ChunkPlanArgs {
    int off[5], cnt[5], slots[5], cap[5], qmin[5], qn[5];
};
// Sum over the CTA (all threads call; w: 32 values of scratch, the caller's again on return), the same on
// every thread.
__device__ int block_sum(int v, int* w) {
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarp = blockDim.x >> 5;
    v = __reduce_add_sync(0xffffffffu, v);
    if (lane == 0) w[warp] = v;
    __syncthreads();
    const int x = lane < nwarp ? w[lane] : 0;
    __syncthreads();
    return __reduce_add_sync(0xffffffffu, x);
}
__global__ void k_chunk_plan(const int32_t* order, int n, const int64_t* inst_off, const int64_t* q_off,
                             const int* plan, ChunkPlanArgs a, int* chunk_q, int* chunk_off) {
    __shared__ int wsum[32];
    __shared__ int carry;
    const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, nwarp = blockDim.x >> 5;
    if (tid == 0) carry = 0;
    for (int bk = 0; bk < 5; ++bk) {
        const int off = plan ? plan[5 + bk] : a.off[bk], cnt = plan ? plan[bk] : a.cnt[bk];
        const int cap = a.cap[bk], qn = a.qn[bk];
        int qc = cap;
        if (cnt > 0 && a.qmin[bk] > 0) {
            const long long most = (cnt > a.slots[bk] ? (long long)cnt : 0) + a.slots[bk];
            int n0[4], q0[4];  // this thread's first instances, read once
#pragma unroll
            for (int r = 0; r < 4; ++r) {
                const int k = tid + r * blockDim.x;
                n0[r] = q0[r] = 0;
                if (k < cnt) {
                    const int I = order[off + k];
                    n0[r] = (int)(inst_off[I + 1] - inst_off[I]);
                    q0[r] = (int)min((long long)INT32_MAX, (long long)(q_off[I + 1] - q_off[I]));
                }
            }
            auto chunks_at = [&](long long qs) {  // work items beyond one per instance
                int v = 0;
#pragma unroll
                for (int r = 0; r < 4; ++r) {
                    const unsigned q = (unsigned)min((long long)INT32_MAX, chunk_len(qs, qn, n0[r], cap));
                    if ((unsigned)q0[r] > q) v += ((unsigned)q0[r] - 1) / q;
                }
                for (int k = tid + 4 * blockDim.x; k < cnt; k += blockDim.x) {
                    const int I = order[off + k];
                    const long long nq = q_off[I + 1] - q_off[I], q = chunk_len(qs, qn, inst_off[I + 1] - inst_off[I], cap);
                    if (nq > q) v += (int)((nq - 1) / q);
                }
                return cnt + (long long)block_sum(v, wsum);
            };
            long long lo = a.qmin[bk], hi = lo;
            while (hi < INT32_MAX / 2 && (cap == 0 || hi < cap) && chunks_at(hi) > most) hi *= 2;
            if (hi > lo) {
                lo = hi / 2;  // too many chunks at lo, few enough at hi
                while (hi - lo > max(1ll, lo / 16)) {
                    const long long mid = (lo + hi) / 2;
                    if (chunks_at(mid) > most)
                        lo = mid;
                    else
                        hi = mid;
                }
            }
            qc = qc > 0 ? (int)min((long long)qc, hi) : (int)hi;
        }
        if (tid == 0) chunk_q[bk] = qc;
        // exclusive scan of the chunk counts, continuing the running total
        for (int b0 = 0; b0 < cnt; b0 += blockDim.x) {
            const int k = b0 + tid;
            int v = 0;
            if (k < cnt) {
                const int I = order[off + k];
                const int64_t nq = q_off[I + 1] - q_off[I];
                const long long q = chunk_len(qc, qn, inst_off[I + 1] - inst_off[I], cap);
                v = qc > 0 ? (int)max(1ll, (nq + q - 1) / q) : 1;
            }
            int x = v;
#pragma unroll
            for (int o = 1; o < 32; o <<= 1) {
                const int y = __shfl_up_sync(0xffffffffu, x, o);
                if (lane >= o) x += y;
            }
            if (lane == 31) wsum[warp] = x;
            __syncthreads();
            if (warp == 0) {
                int t = lane < nwarp ? wsum[lane] : 0;
#pragma unroll
                for (int o = 1; o < 32; o <<= 1) {
                    const int y = __shfl_up_sync(0xffffffffu, t, o);
                    if (lane >= o) t += y;
                }
                wsum[lane] = t;
            }
            __syncthreads();
            const int excl = carry + (warp > 0 ? wsum[warp - 1] : 0) + x - v;
            if (k < cnt) chunk_off[off + k] = excl;
            __syncthreads();
            if (tid == blockDim.x - 1) carry = excl + v;
            __syncthreads();
        }
    }
    if (tid == 0) chunk_off[n] = carry;
}

__global__ void k_reverse_i32(const int32_t* in, int32_t* out, int n) {
    int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i < n) out[i] = in[n - 1 - i];
}

// A workspace allocation failed: record it in the error word and launch nothing else.
int alloc_failed(int* err_dev, cudaStream_t st) {
    cudaGetLastError();
    k_or_err<<<1, 1, 0, st>>>(err_dev, kErrAlloc);
    note_launch();
    return -2;
}

}  // namespace

// One persistent launch of k_solve over instances in the given order with caller-provided
// scratch (no allocation): A in shared memory (npad <= 224), variance columns in ws_v
// (max_grid * npad * threads doubles), work counter *counter zeroed by the caller.
int solve_launch_static(const SolveBatch& b, const DevParams& P, int* err_dev, int npad, int threads, int max_grid,
                        int* counter, const int32_t* order, double* ws_v, cudaStream_t st) {
    SolveCtx c;
    c.plan = nullptr;
    c.bucket = 0;
    c.ws_e = nullptr;
    c.ws_e_stride = 0;
    c.b = b;
    c.P = P;
    c.err = err_dev;
    c.counter = counter;
    c.order = order;
    c.inst_base = 0;
    c.n_work = (int)b.n_inst;
    c.npad = npad;
    c.a_in_smem = 1;
    c.stage_panel = 1;
    c.ws_a = nullptr;
    c.ws_a_stride = 0;
    const size_t shm = smem_bytes(npad, 1, 0, 1, b.Xi != nullptr);
    if (cudaFuncSetAttribute(k_solve<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm) != cudaSuccess)
        return -1;
    int dev = 0, n_sm = 0, per_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_solve<false>, threads, shm);
    const int grid = (int)std::min<int64_t>(std::min<int64_t>(b.n_inst, (int64_t)n_sm * std::max(per_sm, 1)), max_grid);
    c.ws_v_stride = (int64_t)npad * threads;
    c.ws_v = ws_v;
    k_solve<false><<<grid, threads, shm, st>>>(c);
    note_launch();
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

namespace {

using SolveKernel = void (*)(SolveCtx);

// Launch shape of bucket i (cnt instances, `queries` in all) in the plain kernels, unless one was chosen
// (autotuner, vgp_set_launch):
// * N > 224, more than eight instances per SM: three CTAs of 256 threads per SM and no panel staging,
//   so that one's diagonal tiles and barriers overlap the others' updates (2190 instances of
//   about 400 points: 104 -> 96 ms).  With fewer, the last round of instances can cost more than the
//   overlap gains (677 instances: 51 -> 75 ms), and the default's 512 threads on one instance stay.
//   Measured on 152 SMs, mean only: sizes spread over 225..1024, 608 instances 71 -> 80 ms, 912 104 -> 99,
//   1217 130 -> 125, 3000 337 -> 319; equal sizes gain 2 (1000 points) to 26 % (230) from 304 to 3000
//   instances, at 1217 and above 3 to 26.
// * 33 to 64 points, heavy evaluation, few instances with 512 queries or more each: 256 threads, so
//   the chunks are twice as long and fewer of them refit the instance (159 leaves of a frame, 384k
//   voxels: 5.2 -> 3.9 ms; but 4803 instances with 64 queries each: 3.6 -> 4.0 ms).  Measured at 36 and 64
//   points with variance: from 512 to 2500 queries each, 20 to 304 instances take 0.76 to 1.02 of
//   the time; at 128, 456 take 1.1.
struct BucketShape {
    int threads, per_sm, stage;
};
// Bucket i was launched with this shape (per_sm: the cap on CTAs per SM, 0: none).
void note_shape(SolveStats* stats, int i, int threads, int per_sm, int stage) {
    if (!stats) return;
    stats->cfg.threads[i] = threads;
    stats->cfg.per_sm[i] = per_sm;
    if (i == 0) stats->cfg.stage_panel = stage;
}
BucketShape bucket_shape(const SolveConfig& cfg, int i, int64_t cnt, int n_sm, bool heavy, int64_t queries) {
    BucketShape b{cfg.threads[i], cfg.per_sm[i], cfg.stage_panel};
    if (cfg.chosen[i]) return b;
    if (i == 0 && cnt > 8 * n_sm) b = {256, 3, 0};
    if (i == 3 && heavy && cnt <= 2 * n_sm && queries >= 512 * cnt) b.threads = 256;
    return b;
}

SolveKernel pick_solve(bool props, bool emu, bool group = false) {
    if (emu && group) return props ? k_solve_emu<true, true> : k_solve_emu<false, true>;
    if (props) return emu ? k_solve_emu<true, false> : k_solve<true>;
    return emu ? k_solve_emu<false, false> : k_solve<false>;
}

// seven bf16 slices of a block's columns, the row scale, one row of diagonal-tile inverses, and an
// appended query row's diagonal entry
constexpr int64_t kEmuBytesPerRow = 7 * 8 * kEB * 2 + 8 + 64 + 8;

// Words of a matrix of `rows` rows in a CTA's workspace (rows: a multiple of 8).
int64_t matrix_words(bool emu, int rows) { return emu ? n_blocks(rows) * 1024 : n_tiles(rows / 8) * 64; }

// Chunk planning of launch i (cnt instances, resident CTAs per SM, threads each): the rule for its chunks
// and the CTAs to spread it over, all resident ones, but for plain launches with variance, whose FP64 pipe one
// warp per sub-partition nearly fills: 16 warps per SM are enough, and more would only refit.
void chunk_args(const SolveBatch& b, int i, int cnt, int n_sm, int per_sm, int threads, bool emu, ChunkPlanArgs& a) {
    const bool heavy = b.want_var || b.nprop > 0;
    const ChunkRule r = chunk_rule(heavy, b.want_var, emu);
    a.cnt[i] = cnt;
    a.cap[i] = r.cap;
    a.slots[i] = n_sm * (emu || !heavy ? per_sm : std::min(per_sm, std::max(1, 512 / threads)));
    a.qmin[i] = r.qmin;
    a.qn[i] = r.qn;
}

// The emulated kernel's shared memory (about 100 KB at N = 1024) fits twice per SM only in the
// largest shared-memory configuration; ask for it (a preference, so a failure is harmless).
template <class Kernel>
void set_emu_carveout(Kernel k) {
    if (cudaFuncSetAttribute(k, cudaFuncAttributePreferredSharedMemoryCarveout, (int)cudaSharedmemCarveoutMaxShared) !=
        cudaSuccess)
        cudaGetLastError();
}

// Stands in for the emulated kernel in resident_clusters.
__global__ void k_no_tensor_memory() {}

// Clusters of n CTAs that run at once, an emulated CTA's shared memory each: fewer than the SMs' CTAs over n,
// for a cluster stays within a part of the GPU (38 would fill 152 SMs at n = 8, 36 run; 74 of 76 at
// n = 4).  0 where no such cluster can run.  The calculator counts one CTA per SM for a kernel with tensor
// memory (see emu_ctas_per_sm), so it is asked about one without; shared memory allows two of
// either.
int resident_clusters(int n, int threads, size_t shm) {
    cudaLaunchAttribute at{};
    at.id = cudaLaunchAttributeClusterDimension;
    at.val.clusterDim.x = n;
    at.val.clusterDim.y = at.val.clusterDim.z = 1;
    cudaLaunchConfig_t lc{};
    lc.gridDim = dim3(n);
    lc.blockDim = dim3(threads);
    lc.dynamicSmemBytes = shm;
    lc.attrs = &at;
    lc.numAttrs = 1;
    int clusters = 0;
    set_emu_carveout(k_no_tensor_memory);
    if (cudaFuncSetAttribute(k_no_tensor_memory, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm) != cudaSuccess ||
        cudaOccupancyMaxActiveClusters(&clusters, k_no_tensor_memory, &lc) != cudaSuccess) {
        cudaGetLastError();
        return 0;
    }
    return clusters;
}

// CTAs that work on an instance together (a cluster) in an emulated launch of at most `items` work
// items (h[N] + more[N] on instances of N points, nmax the largest), on `slots` resident CTAs, up to 8: as
// many as have all items resident, or as end no later by eights (fours) in two rounds than by fours
// (twos) in one.
// K, the rows below and the trailing tiles are shared out, the diagonal blocks and the solves
// are not, and a block of 32 columns costs three cluster barriers; below 128 points nothing
// is left to share.  Two rounds: the items beyond the resident clusters follow the smallest of the first
// round (largest first).  An instance's time goes as N (N + 700) (0.26, 0.41, 0.82, 1.43 and 3.45 ms
// by eights at 130, 224, 400, 640 and 1024 points), and half as many CTAs take 1.0, 1.1, 1.26 and 1.35
// times as long at 400, 500, 640 and 800 points by fours, 1.1 to 1.25 from 500 by twos.  38 instances of
// 130 points: 0.61 ms by eights, 0.41 by fours, 0.47 by one CTA each; of 1024 down to 420: 3.0
// by eights, 4.2 by fours.
int group_ctas(int items, const int* h, const int* more, int nmax, int slots, int threads, size_t shm) {
    if (nmax <= 128) return 1;
    for (int n = 8; n > 1; n /= 2) {
        if ((int64_t)items * n > slots) continue;
        const int fit = resident_clusters(n, threads, shm);
        if (fit >= items) return n;
        if (n == 2 || 2 * fit < items) continue;
        std::vector<int> sizes;  // decreasing
        for (int N = nmax; N > 32; --N) sizes.insert(sizes.end(), h[N] + more[N], N);
        auto cost = [](double N) { return N * (N + 700.0); };
        const double most = cost(nmax) * (1.0 + std::min(n == 8 ? 0.35 : 0.15, std::max(0.0, (nmax - 400) / 1000.0)));
        bool two = true;
        for (int k = 0; fit + k < items; ++k) two = two && cost(sizes[fit - 1 - k]) + cost(sizes[fit + k]) <= most;
        if (two) return n;
    }
    return 1;
}

// Emulated launch with the latent variance: the queries of an instance (up to kBorderQ) are
// appended to its matrix (see fit_instance); the workspaces hold npad + kBorderQ rows, npad a
// multiple of 32 (the matrix is stored in 32x32 blocks).  Otherwise npad rows.
void emu_rows_for(bool emu, const SolveBatch& b, int& npad, int& qmax, int& nrow) {
    qmax = 0;
    if (emu) npad = (npad + 31) & ~31;
    if (emu && b.want_var) qmax = kBorderQ;
    nrow = npad + qmax;
}

// Resident CTAs per SM of the emulated kernel.  The occupancy calculator reports one CTA per SM
// for any kernel that allocates tensor memory, while the SM runs as many as their registers,
// shared memory and tensor memory allow (each CTA holds kEmuTmemCols of the 512 columns), so
// the bound is computed from those resources.
int emu_ctas_per_sm(SolveKernel k, int threads, size_t shm) {
    cudaFuncAttributes fa{};
    int dev = 0, regs_sm = 65536, smem_sm = 0, thr_sm = 2048;
    if (cudaFuncGetAttributes(&fa, k) != cudaSuccess || cudaGetDevice(&dev) != cudaSuccess) {
        cudaGetLastError();
        return 1;
    }
    cudaDeviceGetAttribute(&regs_sm, cudaDevAttrMaxRegistersPerMultiprocessor, dev);
    cudaDeviceGetAttribute(&smem_sm, cudaDevAttrMaxSharedMemoryPerMultiprocessor, dev);
    cudaDeviceGetAttribute(&thr_sm, cudaDevAttrMaxThreadsPerMultiProcessor, dev);
    const int warps = (threads + 31) / 32;
    const int regs_cta = warps * ((fa.numRegs * 32 + 255) & ~255);  // allocated per warp in units of 256
    const size_t smem_cta = shm + fa.sharedSizeBytes + 1024;        // 1 KB reserved per CTA
    int n = kEmuCtasPerSm;
    n = std::min(n, regs_cta > 0 ? regs_sm / regs_cta : n);
    n = std::min(n, (int)(smem_sm / std::max<size_t>(smem_cta, 1)));
    n = std::min(n, thr_sm / std::max(threads, 1));
    return std::max(n, 1);
}

}  // namespace

void graph_cache_destroy(GraphCache& gc) {
    for (auto& e : gc.exec)
        if (e) cudaGraphExecDestroy(e);
    if (gc.e0) cudaEventDestroy(gc.e0);
    if (gc.e1) cudaEventDestroy(gc.e1);
    if (gc.t0) cudaEventDestroy(gc.t0);
    if (gc.t1) cudaEventDestroy(gc.t1);
    if (gc.gs) cudaStreamDestroy(gc.gs);
    gc = GraphCache{};
}

// The map's own stream and the events that join it to a caller's stream, created with the map (or, if
// that failed, by the first call that wants them).
bool graph_cache_ready(GraphCache& gc) {
    if (gc.t1) return true;
    if ((gc.gs || cudaStreamCreateWithFlags(&gc.gs, cudaStreamNonBlocking) == cudaSuccess) &&
        (gc.e0 || cudaEventCreateWithFlags(&gc.e0, cudaEventDisableTiming) == cudaSuccess) &&
        (gc.e1 || cudaEventCreateWithFlags(&gc.e1, cudaEventDisableTiming) == cudaSuccess) &&
        (gc.t0 || cudaEventCreate(&gc.t0) == cudaSuccess) && cudaEventCreate(&gc.t1) == cudaSuccess)
        return true;
    cudaGetLastError();
    return false;
}

namespace {

void add_stats(SolveStats* stats, const std::vector<int>& h) {
    if (!stats) return;
    for (int N = 0; N <= 1024; ++N) {
        int bk = N <= 32 ? 0 : N <= 64 ? 1 : N <= 128 ? 2 : N <= 256 ? 3 : 4;
        stats->bucket_count[bk] += h[N];
        stats->sum_n3 += (double)h[N] * N * N * N;
        stats->sum_n2 += (double)h[N] * N * N;
    }
}

// Graph mode: the whole solve -- size histogram, bucket plan, decreasing-size order and one
// persistent launch per size bucket -- is planned on the device, captured as a CUDA graph on
// the map's private stream and replayed through a cached executable graph (updated in place
// when only the arguments changed).  Launch shapes come from the map's configuration, sized
// for the largest N the batch can hold; CTAs of a bucket with no work exit at once.  Returns
// 0, -1 when a CUDA call failed, or -2 when a workspace could not be allocated (nothing was
// launched; kErrAlloc is set in *err_dev).
int solve_batch_graph(const SolveBatch& b, const DevParams& P, int* err_dev, cudaStream_t st, Arena& ar,
                      SolveStats* stats, bool profile, const SolveConfig* cfg, GraphCache* gc) {
    const int64_t n = b.n_inst;
    if (!graph_cache_ready(*gc)) return -1;
    const bool props = b.nprop > 0;
    const int T = 256;
    int dev = 0, n_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    const int maxn = std::min(std::max(b.max_n, 1), 1024);
    const int lo[5] = {225, 129, 65, 33, 0}, hi[5] = {1024, 224, 128, 64, 32};
    struct Shape {
        int npad, smem_a, stage, threads, grid, qmax, nrow;
        size_t shm;
        bool live, emu;
        SolveKernel kern;
    } sh[5];
    for (int i = 0; i < 5; ++i) {
        Shape& s = sh[i];
        s.live = maxn >= lo[i];
        s.npad = std::max((std::min(hi[i], maxn) + 7) & ~7, 8);
        s.smem_a = i > (P.emulate ? 3 : 0);  // emulated: the buckets above 32 points
        s.emu = !s.smem_a && P.emulate;
        emu_rows_for(s.emu, b, s.npad, s.qmax, s.nrow);
        s.stage = s.smem_a ? 1 : (s.emu ? 0 : cfg->stage_panel);
        s.threads = s.emu ? kEmuThreads : std::min(cfg->threads[i], kPlainThreads);
        s.shm = smem_bytes(s.npad, s.smem_a, b.nprop, s.stage, b.Xi != nullptr, false, s.emu);
        s.kern = pick_solve(props, s.emu);
    }
    // buckets share a kernel: its shared-memory limit is the largest of the live buckets that
    // launch it, set before any occupancy query or captured launch
    for (int i = 0; i < 5; ++i) {
        if (!sh[i].live) continue;
        if (sh[i].emu) set_emu_carveout(sh[i].kern);
        size_t shm_max = 0;
        for (int j = 0; j < 5; ++j)
            if (sh[j].live && sh[j].kern == sh[i].kern) shm_max = std::max(shm_max, sh[j].shm);
        if (cudaFuncSetAttribute(sh[i].kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm_max) != cudaSuccess)
            return -1;
    }
    ChunkPlanArgs ca{};
    for (int i = 0; i < 5; ++i) {
        Shape& s = sh[i];
        if (!s.live) continue;
        int per_sm = 0;
        if (s.emu) {
            per_sm = emu_ctas_per_sm(s.kern, s.threads, s.shm);
        } else {
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, s.kern, s.threads, s.shm);
            per_sm = std::max(per_sm, 1);
            if (cfg->per_sm[i] > 0) per_sm = std::min(per_sm, cfg->per_sm[i]);
        }
        note_shape(stats, i, s.threads, s.emu ? 0 : cfg->per_sm[i], s.stage);
        // no more CTAs, and workspaces, than the batch can have work items in this bucket: its instances
        // and every shortest chunk (without variance and properties splitting rarely pays: no
        // workspace for it)
        chunk_args(b, i, 0, n_sm, per_sm, s.threads, s.emu, ca);
        const int64_t len = chunk_len(ca.qmin[i], ca.qn[i], std::max(lo[i], 1), ca.cap[i]);
        const int64_t items = n + (b.want_var || props ? b.max_pos / len : 0);
        s.grid = (int)std::min<int64_t>(items, (int64_t)n_sm * per_sm);
    }
    // every buffer exists before the capture starts (allocation is not captured); where memory is short,
    // fewer CTAs share the work
    int* hist = (int*)ar.get(Arena::kHist, sizeof(int) * 2 * 1025, st);
    int32_t* order = (int32_t*)ar.get(Arena::kOrder, sizeof(int32_t) * n, st);
    int* counters = (int*)ar.get(Arena::kCounters, sizeof(int) * 16, st);
    int* chunk_off = (int*)ar.get(Arena::kChunks, sizeof(int) * (n + 1 + 5), st);
    if (!hist || !order || !counters || !chunk_off) return alloc_failed(err_dev, st);
    double *ws_a = nullptr, *ws_v = nullptr;
    uint8_t* ws_e = nullptr;
    for (;;) {
        int64_t need_a = 0, need_v = 0, need_e = 0;
        int grid = 0;
        for (const Shape& s : sh) {
            if (!s.live) continue;
            if (!s.smem_a || b.want_var) grid = std::max(grid, s.grid);
            if (!s.smem_a) need_a = std::max<int64_t>(need_a, matrix_words(s.emu, s.nrow) * s.grid);
            if (b.want_var && !s.emu) need_v = std::max<int64_t>(need_v, (int64_t)s.npad * s.threads * s.grid);
            if (s.emu) need_e = std::max<int64_t>(need_e, (int64_t)s.nrow * kEmuBytesPerRow * s.grid);
        }
        ws_a = need_a ? (double*)ar.get(Arena::kWs0, sizeof(double) * need_a, st) : nullptr;
        ws_v = need_v ? (double*)ar.get(Arena::kWs1, sizeof(double) * need_v, st) : nullptr;
        ws_e = need_e ? (uint8_t*)ar.get(Arena::kWs3, need_e, st) : nullptr;
        if (!(need_a && !ws_a) && !(need_v && !ws_v) && !(need_e && !ws_e)) break;
        if (grid <= 1) return alloc_failed(err_dev, st);
        for (Shape& s : sh)
            if (s.live && (!s.smem_a || b.want_var)) s.grid = (s.grid + 1) / 2;
    }
    for (int i = 0; i < 5; ++i)
        if (sh[i].live) ca.slots[i] = std::min(ca.slots[i], sh[i].grid);
    int* chunk_q = chunk_off + n + 1;
    int* cursor = hist + 1025;
    int* plan = counters + 5;
    cudaStream_t gs = gc->gs;
    if (cudaEventRecord(gc->e0, st) != cudaSuccess || cudaStreamWaitEvent(gs, gc->e0, 0) != cudaSuccess) return -1;
    if (cudaStreamBeginCapture(gs, cudaStreamCaptureModeThreadLocal) != cudaSuccess) return -1;
    fill_i32(hist, 0, 1025, gs);
    fill_i32(counters, 0, 5, gs);
    k_hist_n<<<(unsigned)((n + T - 1) / T), T, 0, gs>>>(b.inst_off, b.q_off, n, hist, nullptr, false, false, false);
    note_launch();
    k_plan_buckets<<<1, 32, 0, gs>>>(hist, cursor, plan);
    note_launch();
    k_order_n<<<(unsigned)((n + T - 1) / T), T, 0, gs>>>(b.inst_off, n, cursor, order);
    note_launch();
    k_chunk_plan<<<1, 1024, 0, gs>>>(order, (int)n, b.inst_off, b.q_off, plan, ca, chunk_q, chunk_off);
    note_launch();
    for (int i = 0; i < 5; ++i) {
        const Shape& s = sh[i];
        if (!s.live) continue;
        SolveCtx c;
        c.chunk_off = chunk_off;
        c.chunk_q = chunk_q + i;
        c.chunk_qn = ca.qn[i];
        c.chunk_cap = ca.cap[i];
        c.b = b;
        c.P = P;
        c.err = err_dev;
        c.counter = counters + i;
        c.order = order;
        c.inst_base = 0;
        c.n_work = 0;
        c.plan = plan;
        c.bucket = i;
        c.npad = s.npad;
        c.a_in_smem = s.smem_a;
        c.stage_panel = s.stage;
        c.qmax = s.qmax;
        c.nrow = s.nrow;
        c.ws_a_stride = s.smem_a ? 0 : matrix_words(s.emu, s.nrow);
        c.ws_a = s.smem_a ? nullptr : ws_a;
        c.ws_v_stride = (int64_t)s.npad * s.threads;
        c.ws_v = ws_v;
        c.ws_e_stride = s.emu ? (int64_t)s.nrow * kEmuBytesPerRow : 0;
        c.ws_e = s.emu ? ws_e : nullptr;
        s.kern<<<s.grid, s.threads, s.shm, gs>>>(c);
        note_launch();
    }
    cudaGraph_t graph = nullptr;
    if (cudaStreamEndCapture(gs, &graph) != cudaSuccess || !graph) return -1;
    cudaGraphExec_t& ex = gc->exec[props ? 1 : 0];
    if (ex) {
        cudaGraphExecUpdateResultInfo info;
        if (cudaGraphExecUpdate(ex, graph, &info) != cudaSuccess) {
            cudaGetLastError();
            cudaGraphExecDestroy(ex);
            ex = nullptr;
        }
    }
    if (!ex) {
        if (cudaGraphInstantiate(&ex, graph, 0) != cudaSuccess) {
            ex = nullptr;
            cudaGraphDestroy(graph);
            return -1;
        }
        ++gc->instantiations;
    }
    cudaGraphDestroy(graph);
    if (profile) cudaEventRecord(gc->t0, gs);
    if (cudaGraphLaunch(ex, gs) != cudaSuccess) return -1;
    ++gc->replays;
    if (profile) cudaEventRecord(gc->t1, gs);
    if (cudaEventRecord(gc->e1, gs) != cudaSuccess || cudaStreamWaitEvent(st, gc->e1, 0) != cudaSuccess) return -1;
    // statistics: the size histogram, read once after the solve
    std::vector<int> h(1025);
    cudaMemcpyAsync(h.data(), hist, sizeof(int) * 1025, cudaMemcpyDeviceToHost, st);
    if (cudaStreamSynchronize(st) != cudaSuccess) return -1;
    add_stats(stats, h);
    if (profile && stats) {
        float ms = 0.f;
        cudaEventElapsedTime(&ms, gc->t0, gc->t1);
        stats->t_solve_ms += ms;
    }
    return 0;
}

}  // namespace

int solve_batch(const SolveBatch& b, const DevParams& P, int* err_dev, cudaStream_t st, Arena& ar, SolveStats* stats,
                 const BackwardBatch* bw, bool profile, int launch, const SolveConfig* cfg, GraphCache* gc) {
    const SolveConfig dflt;
    if (!cfg) cfg = &dflt;
    const int64_t n = b.n_inst;
    if (stats) stats->cfg = *cfg;
    if (n <= 0) return 0;
    if (launch == VGP_LAUNCH_GRAPH && !bw && gc) {
        const int rc = solve_batch_graph(b, P, err_dev, st, ar, stats, profile, cfg, gc);
        if (rc == -2) return rc;
        if (rc != 0) {
            // leave the capture stream usable and the error visible to the caller
            cudaGraph_t g = nullptr;
            cudaStreamCaptureStatus cs;
            if (gc->gs && cudaStreamIsCapturing(gc->gs, &cs) == cudaSuccess && cs != cudaStreamCaptureStatusNone)
                cudaStreamEndCapture(gc->gs, &g);
            if (g) cudaGraphDestroy(g);
            cudaGetLastError();
            k_or_err<<<1, 1, 0, st>>>(err_dev, kErrLaunch);
            note_launch();
            return -1;
        }
        return 0;
    }
    // size histogram (and, for chunk planning, each bucket's queries) and decreasing-size order
    const bool heavy = !bw && (b.want_var || b.nprop > 0);
    ChunkPlanArgs ca{};
    const int words = bw ? kHistWords : 2 * kHistWords + 2 * 5;
    int* hist = (int*)ar.get(Arena::kHist, sizeof(int) * (words + 1025), st);
    if (!hist) return alloc_failed(err_dev, st);
    int* cursor = hist + words;
    cudaMemsetAsync(hist, 0, sizeof(int) * words, st);
    const int T = 256;
    k_hist_n<<<(unsigned)((n + T - 1) / T), T, 0, st>>>(b.inst_off, b.q_off, n, hist, bw ? nullptr : hist + kHistWords,
                                                        heavy, b.want_var, P.emulate);
    note_launch();
    std::vector<int> h(words);
    cudaMemcpyAsync(h.data(), hist, sizeof(int) * words, cudaMemcpyDeviceToHost, st);
    cudaStreamSynchronize(st);
    const int* more = h.data() + (bw ? 0 : kHistWords);
    unsigned long long hq[5] = {0, 0, 0, 0, 0};
    if (!bw) std::memcpy(hq, more + kHistWords, sizeof(hq));
    std::vector<int> start(1026, 0);
    for (int i = 0; i < 1025; ++i) start[i + 1] = start[i] + h[i];
    cudaMemcpyAsync(cursor, start.data(), sizeof(int) * 1025, cudaMemcpyHostToDevice, st);
    int32_t* order_inc = (int32_t*)ar.get(Arena::kOrder, sizeof(int32_t) * 2 * n, st);
    if (!order_inc) return alloc_failed(err_dev, st);
    int32_t* order = order_inc + n;
    k_order_n<<<(unsigned)((n + T - 1) / T), T, 0, st>>>(b.inst_off, n, cursor, order_inc);
    note_launch();
    k_reverse_i32<<<(unsigned)((n + T - 1) / T), T, 0, st>>>(order_inc, order, (int)n);
    note_launch();
    add_stats(stats, h);
    int* chunk_off = nullptr;
    int* chunk_q = nullptr;
    cudaEvent_t ev0 = nullptr, ev1 = nullptr;
    if (profile) {
        cudaEventCreate(&ev0);
        cudaEventCreate(&ev1);
        cudaEventRecord(ev0, st);
    }
    // size buckets, largest first: A in global workspace above 224, in shared memory below.  With the
    // emulated updates every instance above 32 points takes the same kernel with the same launch
    // shape (A in global memory; a single 32-column block leaves it nothing to gain below), so they
    // share one launch, largest first: four launches one after the other each ended in a nearly
    // empty last wave (0.6, 1.4, 0.6 ms for a coloured frame's three).
    struct Bucket {
        int lo, hi, smem_a;
    };
    const Bucket plain_buckets[5] = {{225, 1024, 0}, {129, 224, 1}, {65, 128, 1}, {33, 64, 1}, {0, 32, 1}};
    const Bucket emu_buckets[5] = {{33, 1024, 0}, {1, 0, 0}, {1, 0, 0}, {1, 0, 0}, {0, 32, 1}};
    const bool emu_call = P.emulate && !bw;
    const Bucket* buckets = emu_call ? emu_buckets : plain_buckets;
    if (emu_call) {
        hq[0] += hq[1] + hq[2] + hq[3];
        hq[1] = hq[2] = hq[3] = 0;
    }
    int dev = 0, n_sm = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n_sm, cudaDevAttrMultiProcessorCount, dev);
    if (launch == VGP_LAUNCH_PER_INSTANCE && !bw) {
        // the plain comparison form: one launch per instance, in instance order, one CTA each
        // workspaces sized for the largest instance (N <= 1024, at most 512 threads, appended
        // query rows of the emulated kernel); the default shapes, whichever were chosen
        if (stats) stats->cfg = dflt;
        if (P.emulate) note_shape(stats, 0, kEmuThreads, 0, 0);
        constexpr int kRowsMax = 1024 + kBorderQ;
        int* ctr = (int*)ar.get(Arena::kCounters, sizeof(int) * n, st);
        uint8_t* ws_e = P.emulate ? (uint8_t*)ar.get(Arena::kWs3, kRowsMax * kEmuBytesPerRow, st) : nullptr;
        double* ws_a = (double*)ar.get(Arena::kWs0, sizeof(double) * matrix_words(true, kRowsMax), st);
        double* ws_v = b.want_var ? (double*)ar.get(Arena::kWs1, sizeof(double) * 1024 * 512, st) : nullptr;
        if (!ctr || !ws_a || (P.emulate && !ws_e) || (b.want_var && !ws_v)) {
            if (profile) {
                cudaEventDestroy(ev0);
                cudaEventDestroy(ev1);
            }
            return alloc_failed(err_dev, st);
        }
        cudaMemsetAsync(ctr, 0, sizeof(int) * n, st);
        std::vector<int64_t> off(n + 1);
        cudaMemcpyAsync(off.data(), b.inst_off, sizeof(int64_t) * (n + 1), cudaMemcpyDeviceToHost, st);
        cudaStreamSynchronize(st);
        for (int64_t I = 0; I < n; ++I) {
            const int N = (int)(off[I + 1] - off[I]);
            SolveCtx c;
            c.plan = nullptr;
            c.bucket = 0;
            c.ws_e = nullptr;
            c.ws_e_stride = 0;
            c.b = b;
            c.P = P;
            c.err = err_dev;
            c.counter = ctr + I;
            c.order = nullptr;
            c.inst_base = (int)I;
            c.n_work = 1;
            c.npad = std::max((N + 7) & ~7, 8);
            c.a_in_smem = c.npad <= 224;
            const bool emu = !c.a_in_smem && P.emulate;
            emu_rows_for(emu, b, c.npad, c.qmax, c.nrow);
            c.stage_panel = emu ? 0 : 1;
            const int threads = emu ? kEmuThreads : c.npad <= 32 ? 64 : c.npad <= 64 ? 128 : c.npad <= 128 ? 256 : 512;
            const size_t shm = smem_bytes(c.npad, c.a_in_smem, b.nprop, c.stage_panel, b.Xi != nullptr, false, emu);
            auto ks = pick_solve(b.nprop > 0, emu);
            c.ws_e_stride = emu ? (int64_t)c.nrow * kEmuBytesPerRow : 0;
            c.ws_e = emu ? ws_e : nullptr;
            cudaFuncSetAttribute(ks, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)shm);
            c.ws_a_stride = c.a_in_smem ? 0 : matrix_words(emu, c.nrow);
            c.ws_a = c.a_in_smem ? nullptr : ws_a;
            c.ws_v_stride = (int64_t)c.npad * threads;
            c.ws_v = ws_v;
            ks<<<1, threads, shm, st>>>(c);
            note_launch();
        }
        if (profile) {
            cudaEventRecord(ev1, st);
            cudaEventSynchronize(ev1);
            float ms = 0.f;
            cudaEventElapsedTime(&ms, ev0, ev1);
            if (stats) stats->t_solve_ms += ms;
            cudaEventDestroy(ev0);
            cudaEventDestroy(ev1);
        }
        return 0;
    }
    // a bucket's launch: shapes, kernel, resident CTAs per SM, clusters and workspaces
    struct Launch {
        int nmax, cnt, npad, qmax, nrow, threads, stage, per_sm, ncta, groups;
        size_t shm;
        int64_t ws_a, ws_v, ws_e;  // strides, per group of CTAs (ws_v: per CTA)
        bool emu;
        SolveKernel kern;
    };
    auto bucket_launch = [&](int i) {
        const Bucket& bk = buckets[i];
        Launch L{};
        for (int N = bk.lo; N <= bk.hi; ++N) {
            L.cnt += h[N];
            if (h[N]) L.nmax = N;
        }
        if (L.cnt == 0) return L;
        const BucketShape bs = bw ? BucketShape{cfg->threads[i], cfg->per_sm[i], cfg->stage_panel}
                                  : bucket_shape(*cfg, i, L.cnt, n_sm, heavy, (int64_t)hq[i]);
        L.npad = std::max((L.nmax + 7) & ~7, 8);
        L.emu = !bw && !bk.smem_a && P.emulate;
        emu_rows_for(L.emu, b, L.npad, L.qmax, L.nrow);
        L.threads = L.emu ? kEmuThreads : std::min(bs.threads, kPlainThreads);
        L.stage = bk.smem_a ? 1 : (L.emu ? 0 : bs.stage);
        L.shm = smem_bytes(L.npad, bk.smem_a, bw ? 0 : b.nprop, L.stage, b.Xi != nullptr, bw != nullptr, L.emu);
        L.kern = bw ? k_backward : pick_solve(b.nprop > 0, L.emu);
        cudaFuncSetAttribute(L.kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L.shm);
        if (L.emu) {
            set_emu_carveout(L.kern);
            L.per_sm = emu_ctas_per_sm(L.kern, L.threads, L.shm);
        } else {
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&L.per_sm, L.kern, L.threads, L.shm);
            L.per_sm = std::max(L.per_sm, 1);
            if (bs.per_sm > 0) L.per_sm = std::min(L.per_sm, bs.per_sm);
        }
        note_shape(stats, i, L.threads, L.emu ? 0 : bs.per_sm, L.stage);
        L.ws_a = bk.smem_a ? 0 : matrix_words(L.emu, L.nrow);
        L.ws_v = b.want_var && !bw && !L.emu ? (int64_t)L.npad * L.threads : 0;
        L.ws_e = L.emu ? (int64_t)L.nrow * kEmuBytesPerRow : 0;
        return L;
    };
    // the launches, the buckets' ranges of the order and the CTAs to spread each over; work items are
    // planned only where some bucket can have more of them than instances
    Launch launches[5];
    bool chunks = false;
    // the smallest instances run on the map's own stream beside the others, where its CTAs fill the SMs
    // that the last of those leave; not while profiling
    bool beside = false;
    for (int i = 0, off = 0; i < 5; ++i) {
        Launch& L = launches[i];
        L = bucket_launch(i);
        ca.off[i] = off;
        off += L.cnt;
        if (L.cnt == 0) continue;
        int items = L.cnt;  // an upper bound of the launch's work items
        if (!bw) {
            chunk_args(b, i, L.cnt, n_sm, L.per_sm, L.threads, L.emu, ca);
            int64_t extra = 0;
            for (int N = buckets[i].lo; N <= buckets[i].hi; ++N) extra += more[N];
            if (ca.cap[i] == 0) extra = std::min<int64_t>(extra, ca.slots[i]);
            // (without a bound, a launch of ten rounds of instances or more has no tail to shorten)
            if (ca.cap[i] == 0 && L.cnt > 10 * ca.slots[i]) {
                ca.qmin[i] = 0;
            } else {
                chunks = chunks || extra > 0;
                items = (int)std::min<int64_t>(INT32_MAX, L.cnt + extra);
            }
        }
        // few emulated work items: clusters of CTAs work on each
        L.ncta = L.emu ? group_ctas(items, h.data(), more, L.nmax, n_sm * L.per_sm, L.threads, L.shm) : 1;
        L.groups = (int)std::min<int64_t>(items, (int64_t)n_sm * L.per_sm / L.ncta);
        if (i == 4) beside = !bw && !profile && L.cnt < n && gc && graph_cache_ready(*gc);
    }
    // Every workspace is obtained before the first launch and before e0: a slot that grew between two
    // launches would give its block back behind the first one's kernel, in the order of st alone, and
    // the allocator may hand that block to a launch on the map's own stream, which waits for
    // nothing after e0.
    // Where memory is short, fewer CTAs share the work.
    int* counters = (int*)ar.get(Arena::kCounters, sizeof(int) * 8, st);
    if (chunks) chunk_off = (int*)ar.get(Arena::kChunks, sizeof(int) * (n + 1 + 5), st);
    double *ws_a = nullptr, *ws_v = nullptr, *ws_v_aside = nullptr;
    uint8_t* ws_e = nullptr;
    bool got = counters && (!chunks || chunk_off);
    while (got) {
        int64_t need_a = 0, need_v = 0, need_v_aside = 0, need_e = 0;
        int groups = 0;
        for (int i = 0; i < 5; ++i) {
            const Launch& L = launches[i];
            if (L.ws_a || L.ws_v) groups = std::max(groups, L.groups);
            need_a = std::max(need_a, L.ws_a * L.groups);
            int64_t& nv = i == 4 && beside ? need_v_aside : need_v;
            nv = std::max(nv, L.ws_v * L.groups);
            need_e = std::max(need_e, L.ws_e * L.groups);
        }
        ws_a = need_a ? (double*)ar.get(Arena::kWs0, sizeof(double) * need_a, st) : nullptr;
        ws_v = need_v ? (double*)ar.get(Arena::kWs1, sizeof(double) * need_v, st) : nullptr;
        ws_v_aside = need_v_aside ? (double*)ar.get(Arena::kWs4, sizeof(double) * need_v_aside, st) : nullptr;
        ws_e = need_e ? (uint8_t*)ar.get(Arena::kWs3, need_e, st) : nullptr;
        got = !(need_a && !ws_a) && !(need_v && !ws_v) && !(need_v_aside && !ws_v_aside) && !(need_e && !ws_e);
        if (got || groups <= 1) break;
        for (Launch& L : launches)
            if (L.ws_a || L.ws_v) L.groups = (L.groups + 1) / 2;
        got = true;
    }
    if (!got) {
        if (profile) {
            cudaEventDestroy(ev0);
            cudaEventDestroy(ev1);
        }
        return alloc_failed(err_dev, st);
    }
    if (chunks) {
        chunk_q = chunk_off + n + 1;
        k_chunk_plan<<<1, 1024, 0, st>>>(order, (int)n, b.inst_off, b.q_off, nullptr, ca, chunk_q, chunk_off);
        note_launch();
    }
    cudaMemsetAsync(counters, 0, sizeof(int) * 8, st);
    beside = beside && cudaEventRecord(gc->e0, st) == cudaSuccess && cudaStreamWaitEvent(gc->gs, gc->e0, 0) == cudaSuccess;
    int done = 0;  // instances already assigned (from the large end)
    for (int bi = 0; bi < 5; ++bi) {
        const Launch& L = launches[bi];
        if (L.cnt == 0) continue;
        const bool aside = beside && bi == 4;
        const cudaStream_t ls = aside ? gc->gs : st;
        SolveCtx c;
        c.plan = nullptr;
        c.bucket = 0;
        c.ws_e = nullptr;
        c.ws_e_stride = 0;
        c.b = b;
        c.P = P;
        c.err = err_dev;
        c.counter = counters + bi;
        c.order = order + done;
        c.inst_base = 0;
        c.n_work = L.cnt;
        c.chunk_off = chunk_off ? chunk_off + done : nullptr;
        c.chunk_q = chunk_q ? chunk_q + bi : nullptr;
        c.chunk_qn = ca.qn[bi];
        c.chunk_cap = ca.cap[bi];
        c.npad = L.npad;
        c.qmax = L.qmax;
        c.nrow = L.nrow;
        c.a_in_smem = buckets[bi].smem_a;
        c.stage_panel = L.stage;
        if (bw) c.bw = *bw;
        c.ncta = L.ncta;
        const int grid = L.groups * L.ncta;
        c.ws_a_stride = L.ws_a;
        c.ws_a = L.ws_a ? ws_a : nullptr;
        c.ws_v_stride = L.ws_v;
        c.ws_v = !L.ws_v ? nullptr : bi == 4 && ws_v_aside ? ws_v_aside : ws_v;
        c.ws_e_stride = L.ws_e;
        c.ws_e = L.ws_e ? ws_e : nullptr;
        // (buckets share kernels, whose limit is that of the bucket shaped last)
        auto kern = L.ncta > 1 ? pick_solve(b.nprop > 0, true, true) : L.kern;
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)L.shm);
        cudaEvent_t b0 = nullptr, b1 = nullptr;
        if (profile) {
            cudaEventCreate(&b0);
            cudaEventCreate(&b1);
            cudaEventRecord(b0, st);
        }
        if (c.ncta == 1) {
            kern<<<grid, L.threads, L.shm, ls>>>(c);
        } else {
            cudaLaunchAttribute at{};
            at.id = cudaLaunchAttributeClusterDimension;
            at.val.clusterDim.x = c.ncta;
            at.val.clusterDim.y = at.val.clusterDim.z = 1;
            cudaLaunchConfig_t lc{};
            lc.gridDim = dim3(grid);
            lc.blockDim = dim3(L.threads);
            lc.dynamicSmemBytes = L.shm;
            lc.stream = ls;
            lc.attrs = &at;
            lc.numAttrs = 1;
            set_emu_carveout(kern);
            cudaLaunchKernelEx(&lc, kern, c);
        }
        note_launch();
        if (aside && (cudaEventRecord(gc->e1, gc->gs) != cudaSuccess || cudaStreamWaitEvent(st, gc->e1, 0) != cudaSuccess)) {
            k_or_err<<<1, 1, 0, st>>>(err_dev, kErrLaunch);
            note_launch();
            return -1;
        }
        if (profile) {
            cudaEventRecord(b1, st);
            cudaEventSynchronize(b1);
            float ms = 0.f;
            cudaEventElapsedTime(&ms, b0, b1);
            if (stats) stats->t_bucket_ms[bi] += ms;
            cudaEventDestroy(b0);
            cudaEventDestroy(b1);
        }
        done += L.cnt;
    }
    if (profile) {
        cudaEventRecord(ev1, st);
        cudaEventSynchronize(ev1);
        float ms = 0.f;
        cudaEventElapsedTime(&ms, ev0, ev1);
        if (stats) stats->t_solve_ms += ms;
        cudaEventDestroy(ev0);
        cudaEventDestroy(ev1);
    }
    return 0;
}

namespace {
// Two pairs of FP32 world coordinates per thread, one in each half of the packed operations (even pairs
// in the lower): the emulated kernel's mixed-precision kernel values in the fixed point.
__global__ void k_kfix_probe(const float* xa, const float* xb, long long* out, int64_t n, DevParams P) {
    __shared__ float2 tab[256];
    for (int j = threadIdx.x; j < 256; j += blockDim.x) {
        float h, l;
        split_pair(P.exp_tab[j], h, l);
        tab[j] = make_float2(h, l);
    }
    __syncthreads();
    const int64_t i = 2 * (blockIdx.x * (int64_t)blockDim.x + threadIdx.x), i1 = i + 1 < n ? i + 1 : i;
    if (i >= n) return;
    F2 a[3];
    float b[6];
    for (int k = 0; k < 3; ++k) {
        a[k] = pair2(xa[3 * i + k], xa[3 * i1 + k]);
        b[k] = xb[3 * i + k];
        b[3 + k] = xb[3 * i1 + k];
    }
    long long k0, k1;
    kfix_ff2(a, b, pair2(P.inv2l2_hi), pair2(P.inv2l2_lo), tab, k0, k1);
    out[i] = k0;
    if (i1 > i) out[i1] = k1;
}
}  // namespace

int debug_kernel_fix(const DevParams& P, const float* xa, const float* xb, int64_t n, long long* out,
                     cudaStream_t st) {
    if (n <= 0) return 0;
    k_kfix_probe<<<(unsigned)((n + 511) / 512), 256, 0, st>>>(xa, xb, out, n, P);
    note_launch();
    return cudaGetLastError() == cudaSuccess ? 0 : -1;
}

}  // namespace vgp
