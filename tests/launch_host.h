#pragma once
#include <set>

namespace fake {
extern std::set<int> refuse;                    // launches (counted from 0) that the device refuses
extern int launches;
extern unsigned cluster, grid_x, grid_y;        // of the last launch
}
