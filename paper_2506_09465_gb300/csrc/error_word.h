// What the device error word means to the caller, in plain C++.
#pragma once

#include "../../include/iugkp.h"
#include "layout.h"

namespace iugkp {

// Status and message of the word's bits (0: IUGKP_OK). A barrier that gave up comes first: the
// iteration counts it leaves behind (-1) look like those of a solve that reached its cap, and set that bit
// too.
inline iugkp_status error_word_status(int e, const char** text) {
  *text = "";
  if (e == 0) return IUGKP_OK;
  if (e & ERR_WAIT) {
    *text = "correction solve: a block waited too long for the others of its team";
    return IUGKP_EDEVICE;
  }
  if (e & ERR_BUDGET) {
    *text = "a particle exceeded the step budget and was dropped";
    return IUGKP_EBUDGET;
  }
  if (e & ERR_PCG) {
    *text = "PCG reached cg_maxit before cg_rtol";
    return IUGKP_ENOCONV;
  }
  *text = e & ERR_DEFER ? "more particles than the replay queue holds needed the FP64 walk (queue overflow)"
                        : "device-side check failed";
  return IUGKP_EDEVICE;
}

// The word after a correction's failure has been reported: the bits of the sweeps stay for their own
// check.
inline int error_word_after_correction(int e) { return e & ~(ERR_WAIT | ERR_PCG); }

}  // namespace iugkp
