// Numbers of the state fields and primitives (see include/sacra2d.h).
#pragma once

namespace sacra {

enum : int {
  fW = 0, fHXX, fHXY, fHXZ, fHYY, fHYZ, fHZZ, fAXX, fAXY, fAXZ, fAYY, fAYZ, fAZZ,
  fKH, fGX, fGY, fGZ, fTH, fAL, fBX, fBY, fBZ, fBBX, fBBY, fBBZ,
  fQD, fQSX, fQSY, fQSZ, fQE
};
enum : int { pRHO = 0, pUX, pUY, pUZ, pP, pEPS };

}  // namespace sacra
