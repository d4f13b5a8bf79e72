// precond_layout.h -- the panel of the preconditioner's blocked elimination (precond.cu).
#pragma once

namespace lfmm {

#define PC_NB 16   // most columns of a block
// Columns of a block whose panel of q rows stays in shared memory: PC_NB within 200 KB, fewer for
// larger neighbourhoods, and 0 (a panel of PC_NB columns in global memory) where not even four fit:
// four leaves with a neighbourhood of 3,280 points take 2.89 s so, 4.38 s with three columns in shared
// memory (4,000 points: 5.06 and 7.67 s), and 3,160 points with four columns 2.88 s.
inline int pc_panel_columns(int q) {
    const int n = 200 * 1024 / (16 * (q > 0 ? q : 1));
    return n >= PC_NB ? PC_NB : n >= 4 ? n : 0;
}

}  // namespace lfmm
