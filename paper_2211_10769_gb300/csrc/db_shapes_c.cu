// db_shapes_c.cu -- tile shapes of the packed database search (db_launch.cuh).
#include "sw.h"
#include "db_launch.cuh"

swgb::DbShape swgb::db_shape_c(int k) {
    switch (k) {
        case 0: return db_shape_ops<29, 8, 16>();
        case 1: return db_shape_ops<32, 8, 16>();
        case 2: return db_shape_ops<32, 16, 32>();
        case 3: return db_shape_ops<29, 16, 32>();
        case 4: return db_shape_ops<24, 16, 32>();
        default: return db_shape_ops<16, 16, 32>();
    }
}
