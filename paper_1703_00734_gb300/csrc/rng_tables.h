// rng_tables.h -- the tables of the device generator's normals (host side: rng_tables.cpp).
#pragma once

namespace bmf {

// Reciprocals and logarithms of 1024 intervals of [1, 2); sine and cosine of 512 steps of a
// quarter turn, as doubles and as float pairs.
constexpr int kLogHalf = 424;
struct alignas(32) SinCos {
    double s, c;
    float sp[4];    // s and c as pairs
};
struct alignas(16) LogEntry {
    double c, ln;   // reciprocal, -ln c (less ln 2 from kLogHalf on)
};
struct GenTables {
    LogEntry lg[1024];
    SinCos sc[512];
};
const GenTables &gen_tables();

}  // namespace bmf
