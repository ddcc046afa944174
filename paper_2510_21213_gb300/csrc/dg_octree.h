// Octree auxiliary mesh (Sec. 6.2): connectivity, the operator's 1-D tables
// and the operator launcher (dg_octree.cu), shared with the octree solver
// (dg_octree_solve.cu).
#pragma once

#include <stdint.h>

#include "dg_internal.h"

namespace dg {

// 1-D tables of the octree operator for one degree (n1 nodes per axis)
struct OctTables {
  double w[MAXN1];               // GL weights
  double S[MAXN1 * MAXN1];       // sum_q wq l_a'(xq) l_b'(xq)
  double Lh[2][MAXN1 * MAXN1];   // [c][i][a] l_a((xq_i + 2c - 1) / 2): a larger leaf's basis on half c
  double Le[2][MAXN1];           // l_a(-1), l_a(+1)
  double dLe[2][MAXN1];          // l_a'(-1), l_a'(+1)
};

void octree_tables(int n1, OctTables& T);

// Face connectivity of a leaf set ([E][4] level, ix, iy, iz); per leaf and face
// f = 2 d + side: kind 0 boundary, 1 same-size neighbour, 2 larger neighbour
// (pos: this face's quarter of it), 3 four smaller neighbours (nb[4]). False
// for a bad mesh, a leaf set that is not a partition, or one not 2:1 balanced.
bool octree_faces(const dg_mesh_desc* root, const int32_t* leaves, int32_t n_leaves, int32_t* kind, int32_t* nb,
                  int32_t* pos);

// Hanging faces: rec [nI][6] = larger leaf, its face, the four smaller leaves (by
// quarter); hslot [E][6] = 5 i for the larger side of face i, 5 i + 1 + j for the
// j-th smaller side, -1 where a face does not hang
void octree_hanging(const int32_t* kind, const int32_t* nb, int E, std::vector<int>& rec, std::vector<int>& hslot);

// length factors of the operator, [E][6]: h_t0 h_t1 / (2 h_d), then 1 (penalty
// form 0) or 1 / h_d; hq [E][3] leaf sizes
void octree_factors(const double* hq, int E, int pform, std::vector<double>& fac);

// values that one source's hanging fluxes take
inline size_t octree_hang_elems(int n1, int nI) { return 10 * (size_t)nI * n1 * n1; }

// the mesh on the device: connectivity as octree_faces, fac, hslot and rec as above
struct OctMesh {
  int E;
  const int *kind, *nb;
  const double* fac;
  const int *hslot, *rec;
  int nI;
};

// out[k] = A u[k] (rin null) or rin[k] - A u[k] for the sources k = act[0..nact) (act null: k = 0..nact),
// u and out [.][E][n1^3]; V = double or float (the fields and the arithmetic);
// gbuf: scratch of gelems values, at least octree_hang_elems (sources go through
// in chunks that fit)
template <typename V>
cudaError_t launch_octree_apply(int n1, const OctTables& T, const OctMesh& m, double eps, const V* u, V* out,
                                const V* rin, const int* act, int nact, V* gbuf, long long gelems, cudaStream_t s);

// out[k] = A u[k], k = 0 .. B - 1 (B at most 65535), in one launch and without scratch: the same bits
cudaError_t launch_octree_direct(int n1, const OctTables& T, const OctMesh& m, double eps, const double* u, double* out,
                                 int B, cudaStream_t s);

}  // namespace dg
