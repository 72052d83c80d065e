// Exact-split ("limb") matrix products on the tensor cores, and the local
// convolutions built on them (tiers FP64 and DF).  See limb_gemm.cu and
// limb_conv.cu; the index maps here are shared by host and device code.
//
// A number x with |x| < 2^e is held as the integer X = rint(x 2^(55-e)) in seven
// balanced base-256 digits d_0 .. d_6 (X = sum d_i 256^(6-i), |d_i| <= 128), each
// of them an FP16 value.  A product of two such matrices is
// 28 FP16 products D_l = sum_{i+j=l} A_i B_j, l < 7, whose FP32 accumulators
// hold whole numbers: with chunks of kLimbChunk x 16 <= 256 terms every partial
// sum stays below 2^24 (level l: at most (l+1) 256 2^14 in the worst case, and
// half of that for the digits a table really has), so nothing is rounded in
// them; the levels l >= 7 left out weigh 2^-56 of the leading one.  What is
// left is one rounding when the sum becomes FP64, against the rounding of each
// of the many steps of an FP64 transform.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <memory>

namespace mlc {

constexpr int kLimbs = 7;                    // digits per number
constexpr int kLimbLevels = 7;               // accumulators: digit pairs with i + j = level
constexpr int kLimbM = 128;                  // table rows per tile
constexpr int kLimbN = 64;                   // columns (patches) per tile
constexpr int kLimbChunk = 16;               // k-steps (of 16) between reads of the accumulators
constexpr int kLimbABlk = kLimbM * 16 * 2;   // bytes of one digit of a (tile, k-step) of the table
constexpr int kLimbBBlk = kLimbN * 16 * 2;   // the same of the columns
constexpr int kLimbAStep = kLimbs * kLimbABlk;
constexpr int kLimbBStep = kLimbs * kLimbBBlk;
constexpr int kLimbMaxParts = 8;

// One block of a block-diagonal product: rows x K of the table by K x columns.
struct LimbPart {
    const unsigned char *A;  // digits: [row tile][k-step][digit][canonical core matrices]
    const double *rf;        // row factors 2^(e_row - 62) (rows padded to the tile)
    long b_off;              // bytes, per column tile, before this part in the column image
    long v_off;              // rows of the parts before this one
    int kst;                 // k-steps of 16
    int rows, tiles;         // rows and row tiles
    int tile0;               // first work tile of this part (tiles x column tiles each)
};

// V[part][column][row] = rf[row] cf[part][column] sum_k A[row][k] B[k][column].
struct LimbJob {
    LimbPart part[kLimbMaxParts];
    int nparts;
    const unsigned char *B;  // digits of the columns: [part][column tile][k-step][digit][...]
    const double *cf;        // column factors, [part][cols_pad]
    double *V;               // [part][column][row of the part]
    int cols, ctiles;        // columns and column tiles
    int ntiles;              // work tiles of all parts
    int wait_tries;          // limit of the bounded waits
    int skip_copy;           // test hook: issue no copies, so the bounded waits run out
};

struct Items;
// One launch of the product; a wait that runs out marks the items of its
// columns in their plans' error words.
cudaError_t launch_limb_gemm(const LimbJob &job, const Items &it, cudaStream_t st);
void configure_limb();

// Byte offset of the 8 digits (of one limb) of row `r`, k in [8 q, 8 q + 8) in
// an operand tile of `blk` bytes per digit and k-step: core matrices of 8 rows
// x 16 bytes, the two of a k-step next to each other, rows in groups of 8.
__host__ __device__ inline long limb_chunk_off(int r, int q, int blk) {
    return (long)(q >> 1) * (kLimbs * (long)blk) + (r >> 3) * 256 + (q & 1) * 128 + (r & 7) * 16;
}

// ---- parity classes ---------------------------------------------------------
// The local field of a patch is a convolution with a kernel that is even along
// each axis, over inputs and outputs that are symmetric about the patch centre.
// Folding both into even and odd parts along each axis splits the operator into
// eight blocks (classes, bit 2 - d set: odd along axis d), an eighth of the
// arithmetic in all.  The library's kernel is also the same along the three
// axes, so a class shares the table of its axis permutation with the even axes
// first (classes 0, 1, 3 and 7): axis i of the table is axis limb_perm of the
// class.  A caller-given kernel need not be, and keeps eight tables.
__host__ __device__ constexpr int limb_perm(bool share, int c, int i) {
    constexpr int p[8][3] = {{0, 1, 2}, {0, 1, 2}, {0, 2, 1}, {0, 1, 2}, {1, 2, 0}, {1, 0, 2}, {2, 0, 1}, {0, 1, 2}};
    return share ? p[c][i] : i;
}
__host__ __device__ constexpr bool limb_odd(int c, int d) { return (c >> (2 - d)) & 1; }
__host__ __device__ constexpr int limb_table(bool share, int c) {
    constexpr int t[8] = {0, 1, 1, 3, 1, 3, 3, 7};
    return share ? t[c] : c;
}

// Planes of one kind (face planes, or the planes one node off them): those in
// the lower half are computed, each with its mirror image.
struct LimbPlanes {
    int nrep;
    int c[24];               // normal coordinate
    int slot[24], mslot[24]; // plane slot within its axis of the output, and the mirror image's
    int per_axis;            // slots per axis
};

// Geometry of the folded local convolution of one patch.  Rows of a table, in
// order: the coarse lattice, then per axis the face planes, then per axis the
// off-face planes; in-plane axes in increasing order.
struct LimbConvGeom {
    int n, s, ga, nc, wa;
    int hin[2];      // input reps along an axis: even n/2 + 1, odd n/2
    int hl[2];       // lattice reps, even (the centre included) and odd
    int hp[2];       // in-plane reps
    LimbPlanes face, off;
    bool share;                    // classes share tables up to axis permutations
    int K[8], kst[8], rows[8], tiles[8];  // per table
    long a_off[8], rf_off[8];      // table offsets: bytes, rows (padded)
    long a_bytes, rf_rows;
    long b_step[8], v_step[8];     // per class: bytes per column tile before it, rows before it
    long b_total, v_total;         // of all classes
};

__host__ __device__ inline int limb_lat_rows(const LimbConvGeom &g, int u) {
    return g.hl[limb_odd(u, 0)] * g.hl[limb_odd(u, 1)] * g.hl[limb_odd(u, 2)];
}
// rows of the planes of table axis a (one kind)
__host__ __device__ inline int limb_plane_rows(const LimbConvGeom &g, int u, const LimbPlanes &pl, int a) {
    const int i1 = a == 0 ? 1 : 0, i2 = a == 2 ? 1 : 2;
    return pl.nrep * g.hp[limb_odd(u, i1)] * g.hp[limb_odd(u, i2)];
}
// Row of lattice rep (k0, k1, k2), in table axes.
__host__ __device__ inline int limb_lat_row(const LimbConvGeom &g, int u, int k0, int k1, int k2) {
    return (k0 * g.hl[limb_odd(u, 1)] + k1) * g.hl[limb_odd(u, 2)] + k2;
}
// First row of the planes of a kind (0 face, 1 off) and table axis a.
__host__ __device__ inline int limb_plane_base(const LimbConvGeom &g, int u, int kind, int a) {
    int r = limb_lat_rows(g, u);
    for (int k = 0; k < 2; ++k)
        for (int b = 0; b < 3; ++b) {
            if (k == kind && b == a) return r;
            r += limb_plane_rows(g, u, k ? g.off : g.face, b);
        }
    return r;
}
// Fine coordinates (relative to the patch, table axes) of a row.
__host__ __device__ inline void limb_row_point(const LimbConvGeom &g, int u, int row, int x[3]) {
    const int nl = limb_lat_rows(g, u);
    if (row < nl) {
        const int d2 = g.hl[limb_odd(u, 2)], d1 = g.hl[limb_odd(u, 1)];
        x[2] = -g.s + 4 * (row % d2);
        x[1] = -g.s + 4 * ((row / d2) % d1);
        x[0] = -g.s + 4 * (row / (d2 * d1));
        return;
    }
    row -= nl;
    for (int k = 0; k < 2; ++k)
        for (int a = 0; a < 3; ++a) {
            const LimbPlanes &pl = k ? g.off : g.face;
            const int m = limb_plane_rows(g, u, pl, a);
            if (row < m) {
                const int i1 = a == 0 ? 1 : 0, i2 = a == 2 ? 1 : 2;
                const int d2 = g.hp[limb_odd(u, i2)], d1 = g.hp[limb_odd(u, i1)];
                x[i2] = -g.ga + row % d2;
                x[i1] = -g.ga + (row / d2) % d1;
                x[a] = pl.c[row / (d2 * d1)];
                return;
            }
            row -= m;
        }
    x[0] = x[1] = x[2] = 0;
}
// Input rep (table axes) of column k of a table.
__host__ __device__ inline void limb_col_point(const LimbConvGeom &g, int u, int k, int m[3]) {
    const int d2 = g.hin[limb_odd(u, 2)], d1 = g.hin[limb_odd(u, 1)];
    m[2] = k % d2;
    m[1] = (k / d2) % d1;
    m[0] = k / (d2 * d1);
}

struct Geom;
bool limb_conv_geometry(const Geom &g, bool share, LimbConvGeom &c);

// The folded Green's function tables of one patch geometry and DGF table,
// shared by the plans that use them and freed with the last of them.
struct LimbConvTables {
    LimbConvGeom g;
    unsigned char *A = nullptr;
    double *rf = nullptr;
    ~LimbConvTables();
};
// Tables for a plan's geometry and DGF octant (existing ones are shared).
cudaError_t limb_conv_tables(int device, const Geom &g, bool share, const double *dgf, int dgf_L,
                             std::shared_ptr<LimbConvTables> *out);
inline long limb_ctiles(long items) { return (items + kLimbN - 1) / kLimbN; }
void configure_limb_conv();

}  // namespace mlc
