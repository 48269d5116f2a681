// db_shapes_d.cu -- tile shapes of the packed database search (db_launch.cuh).
#include "sw.h"
#include "db_launch.cuh"

swgb::DbShape swgb::db_shape_d(int k) {
    switch (k) {
        case 0: return db_shape_ops<6, 8, 16>(4690, 161, 199);
        case 1: return db_shape_ops<4, 8, 32>(4190, 130, 159);
        case 2: return db_shape_ops<8, 8, 32>(4940, 171, 191);
        case 3: return db_shape_ops<12, 8, 32>(5340, 227, 250);
        case 4: return db_shape_ops<16, 8, 32>(5540, 268, 291);
        case 5: return db_shape_ops<24, 8, 32>(5620, 370, 377);
        case 6: return db_shape_ops<32, 8, 32>(5690, 464, 471);
        default: return db_shape_ops<12, 8, 16>(5320, 234, 257);
    }
}
