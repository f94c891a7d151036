// occri_chi.cuh -- tables and buffer of the plan's Bloch AOs (occri_chi.cu), as the products
// with them see them.
#pragma once

#include <vector>

#include "occri_internal.h"

namespace occri {

// One shell in slot order.
struct ChiShell {
  double alpha_d, rcut2_d;
  float alpha, alpha_lo, rcut2;
  int l, slot, orig, exact;   // first slot within the atom; index in the basis; FP32 exponents
};

// A contraction's work items for the blocks of one chunk and the first of its rows_of entries.
struct ChiItems {
  int item0 = 0, nitems = 0, row_of0 = 0;
};

// Blocks [b0, b1): one filling of the chi buffer. Items of the tensor cores' contraction (plans
// that run it) and of the CUDA cores', which the adjoint takes in every plan.
struct ChiChunk {
  int b0 = 0, b1 = 0;
  ChiItems tc, con;
};

struct ChiTables {
  std::vector<ChiChunk> chunks;
  int nslots = 0;                 // slots of all atoms, each atom's padded to kChiPad
  int ncls = 0, nkp = 0;          // residue classes in use; k-points padded to 8
  int lsm = 0;                    // image records kept in shared memory (0: read from global)
  int ncol = 0, col_rows = 0;     // AOs per transform over classes (0: none), rows of one
  int buf_rows = 0, warps = 0;    // rows of chi_kernel's buffer, warps of its CTAs
  int signs = 0;                  // every phase of the mesh is a sign (axes of one or two points)
  int parts = 1;                  // CTAs per (block, atom) of chi_kernel
  int kslices = 1;                // slices of the k-points that warps take of a narrow shell
  int batch = 0;                  // images per batch of chi_dense_kernel (0: not this mesh)
  int tile = 0;                   // slots per item of the tensor-core contraction, 0 without it
  long long item_pairs = 0;       // pairs of blocks over the tensor-core items
  size_t chi_bytes = 0;
  // device
  ChiShell* shells = nullptr;     // [nshell] per atom, falling screening radius
  int* slot0 = nullptr;           // [natm + 1] first slot of each atom
  int* slot_ao = nullptr;         // [nslots] AO of a slot, or -1 (padding)
  unsigned short* nsh = nullptr;  // [natm][nblk] shells that reach the block
  int* aoff = nullptr;            // [nblk][natm + 1] slots of the block before atom a
  long long* boff = nullptr;      // [nblk] slots of all blocks before this one in its chunk
  unsigned short* t0i = nullptr;  // [natm][nblk] row of the class table (one per distinct T0)
  int* cls = nullptr;             // [T0][nimg] class of T0 + T'
  int* kidx = nullptr;            // [D_1 D_2 D_3] k-point at each mesh position, or -1
  unsigned short* order = nullptr;   // [natm][nblk][lmax] list positions sorted by class
  void* phase = nullptr;          // [ncls][nkp] e^{i k.T} of each class
  int4* items = nullptr;          // contraction: (atom, first slot, first block, blocks)
  int* border = nullptr;          // blocks per (chunk, atom) by falling number of slots
  int2* rows = nullptr;           // runs of blocks: (first item in the chunk, slot groups)
  int2* rows_of = nullptr;        // [chunk][natm] (first run, runs)
  double* part = nullptr;         // [k][item][values] sums of the items
  float* row_scale = nullptr;     // [nslots] tensor-core contraction: FP16 scale of a slot
  size_t part_bytes = 0;
  void* chi = nullptr;            // [block][k][slot][32 points], complex, or real with signs
  void* arena = nullptr;          // the allocation behind the tables
  void* chunk_arena = nullptr;    // that of what depends on the chunks: boff to rows_of, part, chi
  std::vector<int> aoff_h;        // aoff on the host
};

namespace chi {

constexpr int kPad = 4;         // slots per group: chi_kernel pads with zeros, the products
                                // take kPad AOs at a time

struct Params {
  AOParams a;
  const ChiShell* shells;
  const int* slot0;
  const int* slot_ao;
  const unsigned short* nsh;
  const int* aoff;
  const long long* boff;
  const unsigned short* t0i;
  const int* cls;
  const unsigned short* order;
  const void* phase;
  const int4* items;
  const int* border;
  const int2* rows;
  const int2* rows_of;
  double* part;
  const float* row_scale;
  const double* ao_norm;
  const int* kidx;
  int nslots, ncls, nkp, lsm, parts, ncol, col_rows, buf_rows, warps, signs, batch, kslices;
};

Params params(const Plan& p);
// chi of a chunk's blocks into the buffer
template <typename T>
cudaError_t fill(const Plan& p, const Params& q, const ChiChunk& c, cudaStream_t s);

}  // namespace chi
}  // namespace occri
