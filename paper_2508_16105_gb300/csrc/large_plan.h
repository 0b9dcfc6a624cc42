// Gather plan of the CTA-per-cell kernel (large mechanisms).
//
// Built on the host from the packed mechanism image, uploaded once behind it.
// Every quantity the block accumulates over reactions is listed per output, in
// ascending reaction order, so each output is one thread's fixed-order sum:
//   omega_k     = sum_{e in spr[k]} nu_e q_{r_e}                 (also d omega_k / dT)
//   D[k][j]     = A_k + sum_{q in ent(k,j)} coef_q RS[r_q][slot_q]
//   A_k         = sum_{e in row[k]} nu_e allc_{r_e}              (third-body / falloff [M] term, all j)
// A term is one word: the index of its value in RS (low half; the kernel's shared memory
// bounds 9 R far below 65,536) and of its coefficient in a table of the distinct
// coefficients (high half).  Where there are more than 65,536 of them (a thousand reactions
// each with its own efficiencies), an entry of D counts its indices from its own page of the
// table.  The K * K entries of D come by falling number of terms, so that the lanes of a warp
// loop equally long, each as one int2: page, k and j, and the first term.  At 53 species and 325 reactions the lists take 50 KB, which the L1
// beside three CTAs' shared memory holds (83 KB of terms in three arrays did not): 456 cells
// 74.9 -> 70.8 ms, the adjoint's 152 cells 81.1 -> 71.8 ms.
// where RS[r] holds the reaction's per-side derivatives (slots 0-2 forward, 3-5
// reverse), d q / d[M] (slot 6), q (slot 7) and d q / dT (slot 8).
//
// The plan also carries a compact per-reaction table as structure of arrays
// (ln A, b, E/R, sum of net coefficients; one int4 of packed integers), which the
// kernel stages in shared memory so that consecutive threads read consecutive
// reactions.  Packed integers:
//   x: type (bits 0-1) | reversible (bit 2) | nf (bits 3-4) | nb (bits 5-6) |
//      forward orders (2 bits each from bit 8) | reverse orders (2 bits each from bit 14)
//   y: forward species (10 bits each), z: reverse species (10 bits each), w: spare
#pragma once
#include <stdint.h>

namespace rde {

struct PlanHeader {
  int32_t K, R, n_spr, n_con, n_row, n_coef, bytes, pad;
  // byte offsets of the arrays from the start of the plan (each 16-byte aligned)
  int32_t o_spr_ptr, o_spr, o_ent, o_con, o_row_ptr, o_row, o_coef, o_rx;
  // o_rx: the reaction table, one contiguous block of rx_bytes:
  //   lnA[R], b[R], EaR[R], dnu[R] (doubles, R rounded up to an even count), meta[R] (int4)
  int32_t rx_bytes, rx_stride, pad2[2];
};
static_assert(sizeof(PlanHeader) % 16 == 0, "plan header alignment");

constexpr int kPlanPage = 4096;   // coefficients of a page
struct PlanEntry {
  int32_t kj;     // page << 12 | k << 6 | j
  int32_t first;  // its first term; the next entry's `first` ends the list
};

struct PlanView {
  const int32_t* spr_ptr;   // K + 1
  const uint32_t* spr;      // n_spr terms (slot 7; d omega / dT: the next)
  const PlanEntry* ent;     // K * K + 1
  const uint32_t* con;      // n_con terms
  const int32_t* row_ptr;   // K + 1
  const uint32_t* row;      // n_row terms (slot 6)
  const double* coef;       // n_coef distinct coefficients
};

// Doubles per array of the reaction table (R rounded up so the int4 block stays 16-byte aligned).
#if defined(__CUDACC__)
__host__ __device__ __forceinline__
#else
inline
#endif
int plan_rx_stride(int R) { return (R + 1) & ~1; }

#if defined(__CUDACC__)
__host__ __device__ __forceinline__
#else
inline
#endif
int plan_rx_bytes(int R) { return 4 * 8 * plan_rx_stride(R) + 16 * R; }

#if defined(__CUDACC__)
__host__ __device__ __forceinline__
#else
inline
#endif
PlanView plan_view(const unsigned char* plan) {
  const PlanHeader* h = reinterpret_cast<const PlanHeader*>(plan);
  PlanView v;
  v.spr_ptr = reinterpret_cast<const int32_t*>(plan + h->o_spr_ptr);
  v.spr = reinterpret_cast<const uint32_t*>(plan + h->o_spr);
  v.ent = reinterpret_cast<const PlanEntry*>(plan + h->o_ent);
  v.con = reinterpret_cast<const uint32_t*>(plan + h->o_con);
  v.row_ptr = reinterpret_cast<const int32_t*>(plan + h->o_row_ptr);
  v.row = reinterpret_cast<const uint32_t*>(plan + h->o_row);
  v.coef = reinterpret_cast<const double*>(plan + h->o_coef);
  return v;
}

}  // namespace rde
