// Host program over the kernels' index arithmetic (no GPU, no kernel launched):
// prints "ok" or the first thing that is wrong.
#include <cstdio>
#include <cstdlib>
#include <vector>

#include "kernels.cuh"

#define REQUIRE(c, ...)                    \
    do {                                   \
        if (!(c)) {                        \
            std::printf("wrong: %s ", #c); \
            std::printf(__VA_ARGS__);      \
            std::printf("\n");             \
            std::exit(1);                  \
        }                                  \
    } while (0)

// An in-place step of a ragged row of nx cells.  A plane is read by the
// population opposite to the one that writes it: where the writer stores columns
// (x0 + i, x0 + 1 + i), the reader, moving by -i, loads the same.  Every element
// up to the end of the last sector belongs to one thread: no other one reads it
// or writes it.
template <typename T>
void in_place_row(int nx) {
    const int end = lbm::row_end<T, true>(nx);
    for (int i = -1; i <= 1; ++i) {
        std::vector<int> reader(end, -1), writer(end, -1);
        const auto claim = [&](std::vector<int> &who, int x, int t) {
            REQUIRE(x >= 0 && x < end, "nx %d shift %d thread %d column %d", nx, i, t, x);
            REQUIRE(who[x] < 0, "nx %d shift %d column %d threads %d, %d", nx, i, x, who[x], t);
            who[x] = t;
        };
        for (int t = 0; 2 * t < end; ++t) {
            const lbm::PairCols<true, true> X(2 * t, nx);
            const int store[2] = {i == 0 ? X.x0 : i == 1 ? X.x0 + 1 : X.xm,
                                  i == 0 ? X.x0 + 1 : i == 1 ? X.xp : X.x0};
            const int load[2] = {i == 0 ? X.x0 : i == 1 ? X.x1() : X.xm,
                                 i == 0 ? X.x0 + 1 : i == 1 ? X.xp : X.x0};
            for (int k = 0; k < 2; ++k) {
                claim(writer, store[k], t);
                claim(reader, load[k], t);
                if (X.at < nx)  // a cell: the periodic row
                    REQUIRE(store[k] == (X.at + k + i + nx) % nx, "nx %d shift %d thread %d", nx, i,
                            t);
            }
            REQUIRE(X.x0 == X.at && !X.single(), "nx %d thread %d", nx, t);
            REQUIRE(X.field() + 1 < nx && (X.at >= nx || X.field() == X.at), "nx %d thread %d", nx,
                    t);
        }
        REQUIRE(reader == writer, "nx %d shift %d", nx, i);
    }
}

// A two-buffer step, and an adjoint step with its accumulator (a dense field,
// read and written in place): every cell of the field has one owner.
template <typename T>
void two_buffer_row(int nx) {
    const int end = lbm::row_end<T, true>(nx);
    std::vector<int> owner(nx, -1);
    for (int t = 0; 2 * t < end; ++t) {
        const lbm::PairCols<true> X(2 * t, nx);
        REQUIRE(X.field() == X.x0 && X.x0 >= 0 && X.x0 < nx, "nx %d thread %d", nx, t);
        REQUIRE(X.xm == (X.x0 + nx - 1) % nx && X.xp == (X.single() ? 0 : (X.x0 + 2) % nx) &&
                    X.x1() == (X.x0 + 1) % nx,
                "nx %d thread %d", nx, t);
        if (!X.owner()) continue;
        for (int x = X.x0; x < X.x0 + (X.single() ? 1 : 2); ++x) {
            REQUIRE(x < nx && owner[x] < 0, "nx %d column %d thread %d", nx, x, t);
            owner[x] = t;
        }
    }
    for (int x = 0; x < nx; ++x) REQUIRE(owner[x] == x / 2, "nx %d column %d", nx, x);
}

// The last element of a plane, in the form that the dispatch gives the grid
// (ragged()): byte offsets wrap at 2^32.  No memory is touched.
template <typename T>
void last_element(int nx, int ny, int nz, bool want) {
    lbm::Grid g{};
    g.nx = nx;
    g.ny = ny;
    g.nz = nz;
    g.px = (nx + 31) / 32 * 32;
    g.pop = (long long)g.px * ny * nz;
    const bool rag = lbm::ragged<T>(g);
    REQUIRE(rag == want, "%d x %d x %d of %d bytes", nx, ny, nz, int(sizeof(T)));
    T *const plane = reinterpret_cast<T *>(uintptr_t(1) << 40);
    const int e = int(g.pop - 1);
    const T *const at[2] = {rag ? lbm::element<true>(plane, e) : lbm::element<false>(plane, e),
                            rag ? lbm::element<true, true>(plane, e)
                                : lbm::element<false, true>(plane, e)};
    for (const T *p : at)
        REQUIRE(reinterpret_cast<uintptr_t>(p) ==
                    reinterpret_cast<uintptr_t>(plane) + uintptr_t(e) * sizeof(T),
                "%d x %d x %d of %d bytes", nx, ny, nz, int(sizeof(T)));
}

int main() {
    last_element<float>(1024, 1024, 1024, false);  // 2^32 bytes
    last_element<float>(1024, 1024, 1025, true);
    last_element<float>(32, 32768, 1025, true);
    last_element<float>(1536, 1024, 1024, true);
    last_element<float>(1023, 1024, 1024, true);  // ragged by its rows
    last_element<__half>(1024, 1024, 2047, false);
    last_element<__half>(1022, 1024, 2047, true);
    for (int nx = 1; nx <= 600; ++nx) {
        two_buffer_row<float>(nx);
        two_buffer_row<__half>(nx);
    }
    for (int nx = 2; nx <= 600; nx += 2) {
        in_place_row<float>(nx);
        in_place_row<__half>(nx);
    }
    std::printf("ok\n");
    return 0;
}
