// db_shapes_c.cu -- tile shapes of the packed database search (db_launch.cuh).
#include "sw.h"
#include "db_launch.cuh"

swgb::DbShape swgb::db_shape_c(int k) {
    switch (k) {
        case 0: return db_shape_ops<29, 8, 16>(5990, 447, 455);
        case 1: return db_shape_ops<32, 8, 16>(5910, 499, 506);
        case 2: return db_shape_ops<32, 16, 32>(5770, 464, 471);
        case 3: return db_shape_ops<29, 16, 32>(5800, 422, 429);
        case 4: return db_shape_ops<24, 16, 32>(5650, 371, 377);
        default: return db_shape_ops<16, 16, 32>(5490, 259, 274);
    }
}
