// db_shapes_b.cu -- tile shapes of the packed database search (db_launch.cuh).
#include "sw.h"
#include "db_launch.cuh"

swgb::DbShape swgb::db_shape_b(int k) {
    switch (k) {
        case 0: return db_shape_ops<18, 8, 16>(5350, 318, 339);
        case 1: return db_shape_ops<20, 8, 16>(5510, 326, 341);
        case 2: return db_shape_ops<22, 8, 16>(5590, 364, 376);
        case 3: return db_shape_ops<24, 8, 16>(5870, 381, 392);
        default: return db_shape_ops<26, 8, 16>(5730, 396, 410);
    }
}
