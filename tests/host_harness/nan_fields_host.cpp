// Host harness for tests only: the kernel's lower-star core (lower_star.cuh, keys included) over a whole
// grid, as a program that the test builds with the address and bounds checks of the compiler.  argv[1] holds
// nx, ny, nz (int64) and the field (float32 bits); the packed words are written to argv[2].
#include <cstdint>
#include <cstdio>
#include <cstdlib>
#include <vector>

#define __host__
#define __device__
#define __forceinline__ inline
#include "../../paper_2009_03707_gb300/csrc/lower_star.cuh"

using namespace msc::star;

int main(int argc, char** argv) {
    if (argc != 3) return 2;
    std::FILE* in = std::fopen(argv[1], "rb");
    int64_t d[3];
    if (!in || std::fread(d, sizeof(int64_t), 3, in) != 3) return 2;
    const int nx = int(d[0]), ny = int(d[1]), nz = int(d[2]);
    std::vector<float> field(size_t(nx) * ny * nz);
    std::vector<uint32_t> words(field.size(), 0u);
    if (std::fread(field.data(), 4, field.size(), in) != field.size()) return 2;
    std::fclose(in);
    static Tables T;
    for (int p = 0; p < 27; p++) fill_tables(T, p, 3, 9);
    for (int z = 0; z < nz; z++)
        for (int y = 0; y < ny; y++)
            for (int x = 0; x < nx; x++) {
                uint32_t k[27];
                for (int p = 0; p < 27; p++) {
                    const int X = x + pdx(p), Y = y + pdy(p), Z = z + pdz(p);
                    const bool out = X < 0 || Y < 0 || Z < 0 || X >= nx || Y >= ny || Z >= nz;
                    k[p] = out ? 0xFFFFFFFFu : order_key_of(field[size_t(X) + nx * (size_t(Y) + ny * size_t(Z))]);
                }
                auto emit = [&](int p, uint32_t code) {
                    const int dx = pdx(p), dy = pdy(p), dz = pdz(p);
                    const int ox = x - (dx < 0), oy = y - (dy < 0), oz = z - (dz < 0);
                    if (ox < 0 || oy < 0 || oz < 0) {
                        std::fprintf(stderr, "a cell off the grid was paired\n");
                        std::exit(3);
                    }
                    const int slot = (dx != 0) | ((dy != 0) << 1) | ((dz != 0) << 2);
                    words[size_t(ox) + nx * (size_t(oy) + ny * size_t(oz))] |= code << (3 * slot);
                };
                if (!process_lower_star(k, &T, emit)) return 4;  // a cell left unclassified
            }
    for (int z = 0; z < nz; z++)
        for (int y = 0; y < ny; y++)
            for (int x = 0; x < nx; x++)
                for (int s = 0; s < 8; s++)
                    if (((s & 1) && x == nx - 1) || ((s & 2) && y == ny - 1) || ((s & 4) && z == nz - 1))
                        words[size_t(x) + nx * (size_t(y) + ny * size_t(z))] |= 7u << (3 * s);
    std::FILE* out = std::fopen(argv[2], "wb");
    if (!out || std::fwrite(words.data(), 4, words.size(), out) != words.size()) return 2;
    return std::fclose(out) ? 2 : 0;
}
