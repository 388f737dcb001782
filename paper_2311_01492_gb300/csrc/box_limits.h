// Which kernels a box may take, and which sources the adjoint's kernels share out.  Plain
// C++, so that the choices can be checked on the host.
#pragma once

#include <algorithm>

namespace asora {

// Largest box of the kernels that form a cell's offset within its box in 32 bits (the
// batched traces and the adjoint's whole faces): 1290^3 is the last cube below 2^31.
// Beyond it the plain schedule and the adjoint's quadrant kernels, which count in 64 bits.
constexpr int kMaxBox32 = 1290;

// Sources (LPT order) of the adjoint's launches.  Whole faces by warps: every source if the
// recompute may stop at opaque layers (what does not fit is left to the quadrant kernels,
// through a list on the device), else those whose layers all fit.
struct AdjointPlan {
  int face_begin;  // sources from here on: whole faces
  int quads;       // sources before this one: quadrant kernels, of which
  int split;       // those before this one by CTAs, the others by warps
  bool leftover;   // the faces may leave items to the quadrant kernels
};

// faces: whether whole faces pay (and their tables are there); hbig: half-width of the
// widest source; face_hcap: of the widest that a face has room for; hwarp: of the widest
// that a warp takes a quadrant of (0: none); first_fitting(h): first source of half-width
// h or less (h = 0: ns).
template <class FirstFitting>
AdjointPlan adjoint_plan(int ns, int nmax, bool faces, bool exit, int hbig, int face_hcap,
                         int hwarp, const FirstFitting& first_fitting) {
  AdjointPlan p;
  faces = faces && nmax <= kMaxBox32;
  p.face_begin = !faces ? ns : exit ? 0 : first_fitting(face_hcap);
  p.leftover = faces && exit && hbig > face_hcap;
  p.quads = exit && faces ? (p.leftover ? ns : 0) : p.face_begin;
  p.split = std::min(p.quads, first_fitting(hwarp));
  return p;
}

}  // namespace asora
