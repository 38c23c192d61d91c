#pragma once
#include <set>

namespace fake {
extern std::set<int> refuse;                    // launches (counted from 0) that the device refuses
extern int launches;
extern unsigned cluster;                        // blocks in a cluster of the last launch
}
