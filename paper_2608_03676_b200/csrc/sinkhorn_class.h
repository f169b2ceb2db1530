// Host side of the class kernels (sinkhorn_class.cu): what taot_create learns about the cost matrix.
#pragma once

#include <stdint.h>
#include <vector>

struct taot_class_plan {
    int kind = 0;                     // 0 no class kernel applies, 1 dense, 2 tree
    int nc = 0;                       // dense: classes the kernel is built for (2, 4, 8, 16, 32)
    int gpl = 0, npg = 0;             // tree: groups per lane, classes per group
    float tier[3] = {0.0f, 0.0f, 0.0f};   // tree: cost inside a class, inside a group, elsewhere
    std::vector<int> rep;             // [R] first rank of the rank's class
    std::vector<int> slot_rep;        // [slots] first rank of the slot's class, or -1
    std::vector<uint16_t> cls;        // [R] slot of the rank's class
    std::vector<int32_t> off;         // [slots + 1]
    std::vector<uint16_t> list;       // [R] ranks by slot
    std::vector<float> cost;          // dense: [nc][nc]
};

void taot_build_classes(taot_class_plan* out, const float* C, int R);
