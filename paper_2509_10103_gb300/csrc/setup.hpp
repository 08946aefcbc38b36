// Host-side construction of the discrete operators (FP64, computed once per
// context).  Section 2.4 of Keuchel & Avila: Fourier-Galerkin in theta and z,
// high-order finite differences on Chebyshev radial points, influence-matrix
// wall conditions; Eq. 2.3-2.4 for the base flow.
#pragma once

#include <complex>
#include <string>
#include <memory>
#include <utility>
#include <vector>

namespace pnop {

constexpr int kBand = 13;   // stored band per row: columns j-4 .. j+8
constexpr int kLo = 4;      // lower bandwidth
constexpr int kUp = 8;      // upper bandwidth (one-sided wall stencils)
constexpr int kStencil = 9; // finite-difference points per row

struct Dims {
    int nr = 0, M = 0, K = 0;
    int nm = 0, nk = 0;       // 2M+1, K+1
    int nth = 0, nzp = 0;     // physical 3(M+1), 3(K+1)
    double Lz = 0, stretch = 0;
};

struct Physics {
    double Re = 0, Wo = 0, A = 0, dt = 0, tau0 = 0;
};

// Banded LU factor tables are tiled for the device solver: k is grouped in
// tiles of kTileK consecutive values (one tile = the systems of one solver
// block), and within a (matrix, tile) the forward-sweep columns [0, nc1) of
// every row come first, then the backward-sweep columns [nc1, kBand):
//   table[mat][tile][part 0: j][e < nc1][kk] , [part 1: j][e - nc1][kk]
// so a run of consecutive rows of one sweep is one contiguous piece.
constexpr int kTileK = 32;
inline size_t fac_index(int mat, int k, int j, int e, int nr, int ntile, int nc1) {
    const size_t tile = ((size_t)mat * ntile + k / kTileK) * (size_t)nr * kBand * kTileK;
    const size_t in = e < nc1 ? ((size_t)j * nc1 + e) * kTileK
                              : (size_t)nr * nc1 * kTileK + ((size_t)j * (kBand - nc1) + (e - nc1)) * kTileK;
    return tile + in + k % kTileK;
}
constexpr int kNc1Direct = kLo;          // A x = b rows: l (4) | 1/diag, U (9)
constexpr int kNc1Transposed = kUp + 1;  // A^T x = b rows: U^T (8), 1/diag | L^T (4)

// Fixed-point factor table of the integer solver, which takes each system from
// both ends at once.  The rows [0, h) and [h, nr) are eliminated towards h, up
// to the four rows on either side of it; with those eight kept as one block S,
//   A = N M:  N unit (multipliers of the outer rows), M = D U outside (U with a
//   unit diagonal, coupling a row to the rows nearer h) and S in the middle.
// A side counts its rows ("positions") from its end of the grid inwards, in
// chunks of four; the last chunk is its half of the middle, and the inner side's
// positions are shifted so that it is whole (empty positions at the axis).
// The sweeps need, negated and in fixed point (58 fractional bits, kept as a
// signed high and a signed low 32-bit digit), per position four multipliers of
// N or U by row (direct) or by column (transposed).  A (matrix, tile of kTileX
// k) holds, a 16-byte read being two multipliers of one k:
//   side 0 then side 1:  inward, [chunk][4][2][k][2] (positions p-4..p-1);
//     outward, [chunk but the last]: [4][2][k][2] (positions p+1..p+4) and 1/D as
//     [4][k], a 62-bit fixed-point number whose lowest bits make up an exponent,
//     shared by the rows of a chunk but in the first one; the side's half of S^-1 (or
//     its transpose), [4][4][k][2] (own four, then the other side's four, in
//     positions), the third digits of these entries, [4][4][k] (two 32-bit ones of
//     one k each), and the exponent, [k];
//   the wider wall rows, [4][4][k]: columns 5..8 of rows 0..3 of U (direct), rows
//     0..3 of U for columns 5..8 (transposed).
// The wall row of A (Dirichlet or Neumann) is not scaled like the others, so
// column 0 of N is large: it is stored times 2^-shift and its value enters the
// window times 2^shift.  The solver's 64-bit sums need sum |multiplier| <=
// kFxRowSum in every row; on unstretched grids the sums are at most 4.0 (21 to 768
// points, Re 1 to 1e5, dt 1e-5 to 1, lengths 0.5 to 1000); wide one-sided stencils
// of stretched grids can exceed it (62 at stretch 0.1).
constexpr int kTileX = 16;
constexpr int kFxBits = 58;
constexpr double kFxRowSum = 6.0;
// largest backward error by rows of a factorisation that is taken (20 roundings of
// 2^-53; unstretched grids of 21 to 256 points stay below 5e-16 at any Re, dt and
// length; with the inverse of the middle in one double, 7e-15 at length 8 and
// 1e-10 at 1000)
constexpr double kFxBackward = 2e-15;
constexpr int kFxMinRows = 21;    // smaller grids keep the FP64 solver
constexpr int kFxMaxChunks = 96;  // chunks of a side the solver keeps units for (768 rows in all)
constexpr int kFxMid = 49;        // words of a side's middle per k
// Memory that its first writer, one of the threads that fill a table, touches first
// (zeroing 170 MB of tables on one thread took a quarter of a 64x64x256 context's
// factorisation)
template <class T> struct RawAlloc : std::allocator<T> {
    template <class U> struct rebind {
        using other = RawAlloc<U>;
    };
    template <class U> void construct(U* p) { ::new ((void*)p) U; }
    template <class U, class... A> void construct(U* p, A&&... a) { ::new ((void*)p) U(std::forward<A>(a)...); }
};
using RawVec = std::vector<double, RawAlloc<double>>;
struct FixedTable {
    bool ok = false;
    int shift = 0;
    RawVec direct, transposed;
};
struct FxShape {
    int h, chunks[2], pad;  // rows of side 0, chunks of the sides, empty positions of side 1
    size_t in[2], out[2], mid[2], wall, tile;  // offsets in a tile (8-byte words), its size
};
inline FxShape fx_shape(int nr) {
    FxShape f;
    f.h = 4 * ((nr + 4) / 8 > 4 ? (nr + 4) / 8 : 4);
    const int lower = nr - f.h > 0 ? nr - f.h : 0;
    f.chunks[0] = f.h / 4;
    f.chunks[1] = (lower + 3) / 4;
    f.pad = 4 * f.chunks[1] - lower;
    size_t at = 0;
    for (int s = 0; s < 2; ++s) {
        const size_t n = f.chunks[s], outer = n > 0 ? n - 1 : 0;
        f.in[s] = at;
        f.out[s] = f.in[s] + n * 16 * kTileX;
        f.mid[s] = f.out[s] + outer * 20 * kTileX;
        at = f.mid[s] + kFxMid * kTileX;
    }
    f.wall = at;
    f.tile = f.wall + 16 * kTileX;
    return f;
}

// Words of one matrix's table, room for either form (on grids of 21 and 22 points
// the fixed-point one is the longer).
inline size_t factor_words(int nr, int nk) {
    const size_t fp64 = (size_t)((nk + kTileK - 1) / kTileK) * nr * kBand * kTileK;
    const size_t fixed = (size_t)((nk + kTileX - 1) / kTileX) * fx_shape(nr).tile;
    return fp64 > fixed ? fp64 : fixed;
}

// Everything the device needs, laid out for coalesced access across k.
struct HostOps {
    Dims d;
    Physics ph;
    std::vector<double> r, invr, W;            // [nr]
    std::vector<double> D1, D2;                 // [2 parity][nr][kBand], parity 0 even, 1 odd
    std::vector<double> Lb;                     // [M+2][nr][kBand]  D2 + D1/r - m^2/r^2 (no kz^2)
    // Banded factors for the device: fixed-point tables of M+2 Helmholtz
    // matrices (per |m'|, k) and M+1 pressure matrices (per |m|, k), or where a
    // row's multipliers do not fit (ok false) FP64 rows in the tiled layout of
    // fac_index (ntile tiles of k, zeros beyond nk), "lower | 1/diag | upper":
    //   facH/facP  (A x = b):   l_{j,j-4..j-1}, 1/U_jj, U_{j,j+1..j+8}    (nc1 = kNc1Direct)
    //   facHT/facPT (A^T x = b): U_{j-8..j-1,j}, 1/U_jj, L_{j+1..j+4,j}  (nc1 = kNc1Transposed)
    int ntile = 0;
    FixedTable fxH, fxP;
    RawVec facH, facHT, facP, facPT;
    std::vector<double> phi, dphi;              // [M+1][nk][nr] pressure of a unit wall datum, its radial derivative
    std::vector<double> infl;                   // [nm][3][nr][nk] influence response, pre-scaled by -1/delta
    std::vector<double> fluxg;                  // [nr] flux response of mode (0,0)
    double flux_inv = 0;                        // 1 / sum_j W_j g_j
    std::vector<std::complex<double>> Uh, dUh;  // [nr] oscillatory base-flow profiles
    double omega = 0;                           // pulsation angular frequency Wo^2/Re
};

int parity_index(int m);  // 0 when m is even, 1 when odd

// Builds grid, weights and finite differences (Re-independent part).
bool build_grid(HostOps& h, std::string& err);
// Builds base flow, banded LU factors, influence and flux vectors.
// reuse_pressure: keep h.phi and h.dphi, and leave the pressure tables alone, when it
// already has this grid's size (they depend on the grid only, not on Re or dt).
bool build_operators(HostOps& h, std::string& err, bool reuse_pressure = false);

// Bessel J_nu of complex argument by its power series.
std::complex<double> bessel_j(int nu, std::complex<double> z);

// Factors for the orthogonal projection onto admissible fields (no slip,
// discretely solenoidal; Section 2.2 constraints) in the energy inner product.
// For mode (m, k) != (0, 0), with the wall values removed, the constraint
// C x = D_r x_r + (i m / r) x_theta + i k_z x_z = 0 at every r_j gives the
// real symmetric positive definite system
//   S = D_r W^-1 D_r^T + diag((m^2 / r^2 + k_z^2) / W)  (rows j >= 1 for the diagonal),
// D_r = D1 (parity of m + 1) + 1/r over the columns j >= 1, banded with
// half-bandwidth kProjBand.  L holds its banded Cholesky factor per (|m|, k):
// [|m| = 0..M][k][j][e], e = i - j + kProjBand for i = j - kProjBand .. j - 1,
// and e = kProjBand holding 1 / L_jj.
constexpr int kProjBand = 12;
bool build_projection(const HostOps& h, std::vector<double>& L, std::string& err);

// Binomial checkpointing (Section 2.5).
long long binom_beta(int s, long long t);
int revolve_repetitions(long long nsteps, int snaps);
long long revolve_advances(long long nsteps, int snaps);

}  // namespace pnop
