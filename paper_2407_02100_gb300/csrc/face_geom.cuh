// Faces of one colour of the shared-face sweep: numbering, buffer layout and
// node origins, shared by the face and patch kernels of both precisions.
#pragma once
#include "kernels.h"

namespace gmg {

// Patch (i_x, i_y, i_z) of the colour owns
//   x faces fx = i_x, i_x + 1 of X[(i_z c_y + i_y)(c_x + 1) + fx],
//   y faces fy = i_y, i_y + 1 of Y[(i_z (c_y + 1) + fy) c_x + i_x],
//   z faces fz = i_z, i_z + 1 of Z[(fz c_y + i_y) c_x + i_x].
// Each face holds two M x M fields padded to a multiple of 16 bytes
// (face_fields elements); the families start at foff[0..2] elements.
struct FaceGeom {
  long long py, pz;
  int first[3], count[3];
  long long nf[3];
  long long foff[3];
};

// elements (of elem_bytes) of one face's two fields
__host__ __device__ constexpr int face_fields(int k, int elem_bytes) {
  return (2 * (2 * k - 1) * (2 * k - 1) + 16 / elem_bytes - 1) / (16 / elem_bytes) * (16 / elem_bytes);
}

// element offset of the first node of face f of family fam (0 x, 1 y, 2 z):
// the face planes of patch (i_x, i_y, i_z) sit at its closure origin (index
// i) and at the next patch's (index i + 1); in-plane the data start at the
// closure origin (axes the face spans completely) or one node inside it
// (interior rows)
template <int K>
__device__ __forceinline__ long long face_origin(const FaceGeom& fg, int fam, long long f) {
  const int cx = fg.count[0], cy = fg.count[1];
  long long ix, iy, iz;
  if (fam == 0) {
    ix = f % (cx + 1);
    const long long r = f / (cx + 1);
    iy = r % cy;
    iz = r / cy;
  } else if (fam == 1) {
    ix = f % cx;
    const long long r = f / cx;
    iy = r % (cy + 1);
    iz = r / (cy + 1);
  } else {
    ix = f % cx;
    const long long r = f / cx;
    iy = r % cy;
    iz = r / cy;
  }
  const long long X = (fg.first[0] + 2 * ix - 1) * K + (fam == 0 ? 0 : 1);
  const long long Y = (fg.first[1] + 2 * iy - 1) * K + (fam == 2 ? 1 : 0);
  const long long Z = (fg.first[2] + 2 * iz - 1) * K;
  return X + fg.py * Y + fg.pz * Z;
}

inline FaceGeom face_geom(const PatchLaunch& pl, int elem_bytes) {
  FaceGeom fg;
  fg.py = pl.g.py;
  fg.pz = pl.g.pz;
  for (int a = 0; a < 3; ++a) {
    fg.first[a] = pl.first[a];
    fg.count[a] = pl.count[a];
  }
  const long long cx = pl.count[0], cy = pl.count[1], cz = pl.count[2];
  fg.nf[0] = (cx + 1) * cy * cz;
  fg.nf[1] = cx * (cy + 1) * cz;
  fg.nf[2] = cx * cy * (cz + 1);
  const long long fs = face_fields(pl.g.k, elem_bytes);
  fg.foff[0] = 0;
  fg.foff[1] = fg.nf[0] * fs;
  fg.foff[2] = fg.foff[1] + fg.nf[1] * fs;
  return fg;
}

// elements of the face buffer for one colour launch of pl's geometry
inline long long face_buffer_total(const PatchLaunch& pl, int elem_bytes) {
  const FaceGeom fg = face_geom(pl, elem_bytes);
  return (fg.nf[0] + fg.nf[1] + fg.nf[2]) * face_fields(pl.g.k, elem_bytes);
}

}  // namespace gmg
