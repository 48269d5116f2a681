// db_shapes_a.cu -- tile shapes of the packed database search (db_launch.cuh).
#include "sw.h"
#include "db_launch.cuh"

swgb::DbShape swgb::db_shape_a(int k) {
    switch (k) {
        case 0: return db_shape_ops<4, 8, 16>(4150, 147, 207);
        case 1: return db_shape_ops<7, 8, 16>(4690, 173, 209);
        case 2: return db_shape_ops<9, 8, 16>(4930, 209, 244);
        case 3: return db_shape_ops<11, 8, 16>(4820, 270, 307);
        case 4: return db_shape_ops<13, 8, 16>(5310, 241, 265);
        default: return db_shape_ops<16, 8, 16>(5410, 300, 331);
    }
}
