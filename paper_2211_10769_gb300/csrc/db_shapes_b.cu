// db_shapes_b.cu -- tile shapes of the packed database search (db_launch.cuh).
#include "sw.h"
#include "db_launch.cuh"

swgb::DbShape swgb::db_shape_b(int k) {
    switch (k) {
        case 0: return db_shape_ops<18, 8, 16>();
        case 1: return db_shape_ops<20, 8, 16>();
        case 2: return db_shape_ops<22, 8, 16>();
        case 3: return db_shape_ops<24, 8, 16>();
        default: return db_shape_ops<26, 8, 16>();
    }
}
