// Internal layout shared by the host table builder (mech_tables.cpp) and the kernels
// (chem_kernels.cu).  Not part of the public ABI.
#pragma once
#include <array>
#include <cstdint>
#include <string>
#include <vector>

namespace chemgpu {

// Reaction kinds.  Device order: Troe, Lindemann, third-body, elementary, so that lanes of one
// warp pass mostly run the same branch and the pressure-dependent reactions are 0 .. n_pd-1.
enum : int { kElementary = 0, kThirdBody = 1, kLindemann = 2, kTroe = 3 };

// Per-reaction integer record (16 ints).
//   [0..3]  slot species: reactant 0, reactant 1, product 0, product 1 (-1 = empty)
//   [4..7]  distinct slot species, -1 pads
//   [8..11] rows: distinct species k < K-1 with non-zero net coefficient, -1 pads
//   [12..15] net coefficients of those rows
constexpr int kRxInts = 16;

// Per-reaction double record.
//   [0] ln A   [1] b   [2] Ea/Rc (K)   [3..6] net coefficients of the rows (as doubles)
constexpr int kRxDoubles = 7;

// Per fall-off reaction doubles: ln A0, b0, Ea0/Rc, alpha, T3, T1, T2, is_troe, 1/T3, 1/T1
constexpr int kFoDoubles = 10;

// Per species doubles: W, 1/W, Tmid, NASA low a1..a7, NASA high a1..a7
constexpr int kSpDoubles = 17;

// Rows of the per-species table of the fixed-point rate evaluation, [kSpfRows][K] (consecutive
// threads read consecutive words): W, 1/W, Tmid, then kSpfRange rows for each range (low, high), all
// with their constant factors multiplied in on the host:
//   cp/R = sum a_n T^n:                           [0..4]  a1 .. a5
//   h/RT = a1 + T (..) + a6/T:                    [5..8]  a2/2, a3/3, a4/4, a5/5   [9] a6
//   (g/RT) / ln 2 = [10] + [11] log2 T + [12]/T + T ([13] + T ([14] + T ([15] + T [16]))), the first
//     three as the bits of int64: * 2^52, * 2^57, * 2^45 (the largest terms are summed in fixed point)
//   d(cp/R)/dT:                                   [17..19] 2 a3, 3 a4, 4 a5
constexpr int kSpfRange = 20;
constexpr int kSpfRows = 3 + 2 * kSpfRange;

constexpr int kFxIntervalCount = 7;  // temperature intervals tried for fx_T

struct HostMech {
  int K = 0, R = 0, E = 0;
  int n_elem = 0, n_tb = 0, n_fo = 0;  // counts in device order
  std::vector<int> order;              // device reaction index -> file reaction index
  std::vector<double> sp;              // [K][kSpDoubles]
  std::vector<double> rxd;             // [R][kRxDoubles]
  std::vector<int> rxi;                // [R][kRxInts]
  std::vector<int> dnu;                // [R] products minus reactants
  std::vector<double> eff;             // [n_tb + n_fo][K]
  std::vector<double> fo;              // [n_fo][kFoDoubles]
  // species -> (reaction, net coefficient) lists, all K species
  std::vector<int> sr_ptr;             // [K + 1]
  std::vector<int> sr_idx;             // reaction index (device order)
  std::vector<double> sr_nu;           // net coefficient of the species in that reaction
  // Tables of the fixed-point rate evaluation (build_fx_tables).  Logarithms base 2.
  std::vector<double> fx_T;            // {lo, hi}: it takes temperatures inside (equal: none), chosen
                                       // so that every exponent stays inside the fixed-point range
  bool fx_ok = false;                  // every table value but ln A fits its fixed-point format
  // per candidate of fx_T: whether the exponents that do not depend on ln A keep their bounds (-1: not asked yet)
  std::array<int8_t, kFxIntervalCount> fx_thermo_fits;
  std::vector<uint32_t> rx4;           // [R] slot species, one byte each (255 = empty)
  std::vector<int64_t> fxk;            // [3][R] log2 A * 2^52, b * 2^57, Ea/(Rc ln 2) * 2^46
  std::vector<int64_t> fxo;            // [3][n_fo] the same of the low-pressure limit
  std::vector<double> fod;             // [5][n_fo] 1 - alpha, alpha, log2(e)/T3, log2(e)/T1, T2 log2(e)
  std::vector<double> spf;             // [kSpfRows][K]
  std::vector<double> rxd_t;           // [2][R] b, Ea/Rc
  std::vector<double> eff_t;           // [K][n_pd] efficiencies, transposed
  // the same in fixed point, eff * 2^(62 - effe) with effe[r] the exponent that puts the reaction's largest
  // below 1; empty unless every reaction's efficiencies are positive and within a factor of 16
  std::vector<int64_t> effx;           // [K][n_pd]
  std::vector<int> effe;               // [n_pd]
  // species production lists, entry e of species k at [e * K + k]: reaction index in the low half,
  // the top 16 bits of the net coefficient as a double in the high half (small integers have no others)
  std::vector<uint32_t> srx;
  // Jacobian gather plan (mass-action part).  Every Z entry of the species rows (k < K-1, all columns)
  // sums coef * s[src] over its contributions (src an index into the per-reaction scratch).  Entries in
  // order of decreasing list length; the c-th contribution of entry e, where it has one, is at
  // zgx[zgb[c] + e]: src in the low half, the top 16 bits of the coefficient (a small integer) as a
  // double in the high half.
  std::vector<int> zg_dst;             // [(K-1) K] ((row + 1) mod K) * K + (col + 1) mod K
  std::vector<int> zgb;                // [longest list + 12], the last twelve equal
  std::vector<uint32_t> zgx;           // [contributions]
  std::vector<double> mwr;             // [K-1][K-1] -W_k / W_i
  // Efficiency part: for each species row k < K-1, the pressure-dependent reactions in it:
  // (pd index, net coefficient)
  std::vector<int> pr_ptr;             // [K + 1]
  std::vector<int> pr_pd;
  std::vector<double> pr_nu;
  std::vector<int> pr_rows;            // rows with pairs, shortest lists first
  // Column lists (products with J^T): for species column j, the per-reaction scratch indices
  // of dq/dC_j and their reactions
  std::vector<int> cl_ptr;             // [K + 1]
  std::vector<int> cl_src;
  std::vector<int> cl_rx;
};

// Build the tables of the fixed-point rate evaluation from the others.
void build_fx_tables(HostMech& m);
// After a change of ln A: the first row of fxk and fx_T, all that depends on it.
void update_fx_lnA(HostMech& m);

// Parse the mechanism text file; false + message on error.
bool parse_mechanism(const char* path, HostMech& m, std::string& err);

// Device view of the tables (all pointers into one device allocation).
struct DevMech {
  int K, R, N;
  int n_elem, n_tb, n_fo, n_pd;  // fall-off reactions are 0 .. n_fo-1, pressure-dependent 0 .. n_pd-1
  const double* sp;
  const double* rxd;
  const int* rxi;
  const int* dnu;
  const double* eff;
  const double* fo;
  const int* sr_ptr;
  const int* sr_idx;
  const double* sr_nu;
  const int* zg_dst;
  const int* zgb;
  const uint32_t* zgx;
  const double* mwr;
  const int* pr_ptr;
  const int* pr_pd;
  const double* pr_nu;
  const int* pr_rows;
  int n_pairs, n_prows;
  // reaction split of the rate evaluation for groups of 2, 4 and 8 warps (index 1, 2, 3; index 0
  // unused): warp 0 takes reactions [0, split), the other warps [split, R); 0 = interleaved
  int rx_split[4];
  const int* order;  // device reaction index -> file reaction index
  const int* cl_ptr;
  const int* cl_src;
  const int* cl_rx;
  // fixed-point rate evaluation (see HostMech)
  const double* fx_T;  // (in device memory: a captured launch sees chem_set_lnA's change)
  const uint32_t* rx4;
  const int64_t* fxk;
  const int64_t* fxo;
  const double* fod;
  const double* spf;
  const double* rxd_t;
  const double* eff_t;
  const int64_t* effx;  // NULL: none
  const int* effe;
  const uint32_t* srx;
};

}  // namespace chemgpu
