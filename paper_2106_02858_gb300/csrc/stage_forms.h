// The stage-kernel forms and how a handle that is not told one takes its own (host only).
//
// FP32: 0, 1, 2 = one warp per half tile (two threads per tetrahedron) with at least 12, 16, 24
// resident warps per SM; 3, 4 = two warps per half tile with at least 12, 16; 5 = four warps per half
// tile; 6 = tensor-core contractions (tcgen05, 3xTF32).  FP64: 0, 1, 2 = one, two, four warps per half
// tile.
#pragma once

namespace cmcg {

constexpr int STAGE_FORMS_F32 = 7;
constexpr int STAGE_FORM_TC = 6;
constexpr int STAGE_FORMS_F64 = 3;

// Times the forms a handle of this precision and order may take and gives the fastest, *form = -1 if
// the device rejects every one.  `time(f, &us)` times form f (us < 0: rejected) and returns a status;
// us_of[f] is left alone for forms that are not timed.
//
// P3 in FP32 takes the tensor-core form at every size (us per stage, and of the best other form: 48
// tetrahedra 7.6 and 8.8, 1,296 7.9 and 10.1, 10,368 11.3 and 15.2, 48,000 32 and 38), P1 and P2 one of the
// others (P2: 82,944 tetrahedra 31 and 15), and the forms that are timed against each other give the
// same bits: the arithmetic does not depend on what was measured.  Only a device that rejects
// the tensor-core form's launch gives a P3 handle one of the others.
template <typename Time>
int choose_form(bool fp32, int q, double* us_of, int* form, Time&& time) {
  const int first[2] = {fp32 && q == 3 ? STAGE_FORM_TC : 0, 0};
  const int end[2] = {fp32 ? (q == 3 ? STAGE_FORM_TC + 1 : STAGE_FORM_TC) : STAGE_FORMS_F64, fp32 && q == 3 ? STAGE_FORM_TC : 0};
  *form = -1;
  for (int r = 0; r < 2 && *form < 0; ++r)
    for (int f = first[r]; f < end[r]; ++f) {
      const int rc = time(f, &us_of[f]);
      if (rc) return rc;
      if (us_of[f] >= 0 && (*form < 0 || us_of[f] < us_of[*form])) *form = f;
    }
  return 0;
}

}  // namespace cmcg
