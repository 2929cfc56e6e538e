// center_rows.cuh -- which launches of a center graph keep boundary rows (the
// row between two passes, in global memory) and which branch of the graph they
// take.  Plain C++, so the host can check it.
#pragma once

constexpr int kCenterLanes = 8;  // branches of the center graph
constexpr int kRowLanes = 2;     // the first of them have an area of boundary rows each

// npass: the most passes of a query pair in the class.  The bounded kernel
// stores the bottom row of every pass, also of a pair's last or only one.
inline bool center_keeps_rows(int npass, bool bounded) { return bounded || npass > 1; }

// The branch of the class at this launch position: launches of one branch follow
// one another, so two that share an area must share a branch.
inline int center_lane(int order, bool keeps_rows) { return order % (keeps_rows ? kRowLanes : kCenterLanes); }
