"""Rules of the kernels that are plain host and device functions, compiled with nvcc and run on
the CPU: the entries of a tile's run labels that the label of a site reads, and the piece ids
that a tile reserves."""
import subprocess

from paper_1405_1931_gb300 import build, hk

LABELS = r"""
#include <cstdio>
#include <cstdlib>
#include <vector>
#include "hk_device.cuh"
// a tile's run labels: the entries of one row are [first, first + n); any other read is counted
struct Checked {
    int first, n;
    mutable long outside = 0;
    __host__ __device__ int operator[](int i) const {
        if (i < first || i >= first + n) ++outside;
        return 1000 + i;
    }
};
int main() {
    std::vector<unsigned> words = {0u, ~0u, 1u, 1u << 31, 0x55555555u, 0xaaaaaaaau, 0x7ffffffeu, 0x80000001u};
    srand(7);
    for (int i = 0; i < 5000; ++i) words.push_back(((unsigned)rand() << 17) ^ ((unsigned)rand() << 2) ^ (unsigned)rand());
    long outside = 0, wrong = 0;
    for (unsigned m : words)
        for (int first : {0, 1, 37}) {
            const unsigned rs = m & ~(m << 1);
            const Checked lab{first, __builtin_popcount(rs)};
            int run = first - 1;
            for (int x = 0; x < 32; ++x) {
                if ((rs >> x) & 1u) ++run;
                const int want = (m >> x) & 1u ? 1000 + run : -1;
                if (hk::site_label(m, rs, first, hk::le_mask(x), lab) != want) ++wrong;
            }
            outside += lab.outside;
        }
    printf("%ld %ld\n", outside, wrong);
}
"""


PIECES = r"""
#include <cstdio>
#include <cstdlib>
#include <initializer_list>
#include <vector>
#include "hk_device.cuh"
#include "hk_launch.h"
using namespace hk;
template <int TY, int TZ>
TileInfo shape() {
    using SH = TileShape<TY, TZ>;
    return TileInfo{TY, TZ, SH::R, SH::MAXRUNS, SH::FACE_STRIDE, SH::MAX_BOUNDARY};
}
// pieces of one tile of the lattice that touch a face with a neighbour tile
int boundary_pieces(const TileInfo &ti, const int n[3], double p) {
    const int t[3] = {32, ti.ty, ti.tz};
    int e[3];
    for (int a = 0; a < 3; ++a) e[a] = n[a] < t[a] ? n[a] : t[a];
    const int N = e[0] * e[1] * e[2];
    std::vector<int> occ(N), seen(N, 0);
    for (int s = 0; s < N; ++s) {
        const int x = s % e[0], y = s / e[0] % e[1], z = s / e[0] / e[1];
        occ[s] = p < 0 ? (x + y + z) & 1 : rand() < p * RAND_MAX;
    }
    int count = 0;
    for (int s0 = 0; s0 < N; ++s0) {
        if (!occ[s0] || seen[s0]) continue;
        bool touch = false;
        std::vector<int> todo{s0};
        seen[s0] = 1;
        while (!todo.empty()) {
            const int s = todo.back();
            todo.pop_back();
            const int c[3] = {s % e[0], s / e[0] % e[1], s / e[0] / e[1]}, step[3] = {1, e[0], e[0] * e[1]};
            for (int a = 0; a < 3; ++a) {
                if (n[a] > t[a] && (c[a] == 0 || c[a] == e[a] - 1)) touch = true;
                if (c[a] > 0 && occ[s - step[a]] && !seen[s - step[a]]) seen[s - step[a]] = 1, todo.push_back(s - step[a]);
                if (c[a] < e[a] - 1 && occ[s + step[a]] && !seen[s + step[a]]) seen[s + step[a]] = 1, todo.push_back(s + step[a]);
            }
        }
        count += touch;
    }
    return count;
}
int main() {
    long over = 0, wide = 0, refused = 0, small = 0;
    srand(3);
    for (const TileInfo &ti : {shape<8, 8>(), shape<16, 8>(), shape<16, 16>(), shape<32, 8>()}) {
        const int t[3] = {32, ti.ty, ti.tz};
        for (int k = 0; k < 600; ++k) {                   // the bound holds, and is no wider than the shape's
            int n[3];
            for (int a = 0; a < 3; ++a) n[a] = k % 3 ? 1 + rand() % 40 : (rand() & 1 ? 1 + rand() % 3 : t[a] + rand() % 2);
            const int bound = piece_bound(ti, n[0], n[1], n[2]);
            for (double p : {-1.0, 0.3, 0.5}) over += boundary_pieces(ti, n, p) > bound;
            wide += bound > ti.max_boundary || bound % 4;
        }
        const long sites = (1l << 31) - 1;                // every lattice of fewer than 2^31 sites gets ids that fit
        for (long nx : {1, 2, 31, 32, 33, 65, 1024, 32768})
            for (long ny : {1, 2, 7, 8, 9, 15, 16, 17, 32, 33, 34, 1024, 32768, 65535})
                for (int axis = 0; axis < 3; ++axis) {
                    const long n3 = sites / (nx * ny);
                    if (n3 < 1) continue;
                    const long d[3] = {axis == 0 ? n3 : nx, axis == 1 ? n3 : (axis == 0 ? nx : ny), axis == 2 ? n3 : ny};
                    Plan P{};
                    P.ntiles = ((d[0] + 31) / 32) * ((d[1] + ti.ty - 1) / ti.ty) * ((d[2] + ti.tz - 1) / ti.tz);
                    refused += !plan_pieces(ti, P, (int)d[0], (int)d[1], (int)d[2]);
                    small += P.ntiles * ti.max_boundary < (1l << 31) && P.piece_stride != ti.max_boundary;
                }
    }
    printf("%ld %ld %ld %ld\n", over, wide, refused, small);
}
"""


def host_program(tmp_path, source):
    src, exe = tmp_path / "rule.cu", tmp_path / "rule"
    src.write_text(source)
    subprocess.run([build.nvcc(), "-std=c++17", "-O1", *build.ARCH, "-I", build.CSRC, "-o", str(exe), str(src)], check=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout


def test_site_label_reads_its_rows_entries_only(tmp_path):
    assert host_program(tmp_path, LABELS).split() == ["0", "0"]


def test_piece_slices_hold_every_tile_and_ids_fit(tmp_path):
    assert host_program(tmp_path, PIECES).split() == ["0", "0", "0", "0"]


def test_workspace_of_flat_lattices_has_31_bit_piece_ids():
    """12 bytes a piece (parent, key, size) beside what does not depend on the slices."""
    for nx, ny, nz in [(32768, 32768, 1), (1, 27_000_000, 1), (53_760_000, 1, 1), (1, 20800, 20800), (1024, 1024, 1024)]:
        tiles = -(-nx // 32) * -(-ny // 16) * -(-nz // 16)
        rest = tiles * (256 * 4 + 4096 * 2 + 1288 * 2 + 16 + 64 + 4) + -(-nx // 32) * ny * nz + 4 * (ny * nz + 1)
        pieces = (hk.hk_workspace_bytes(nx, ny, nz) - rest) / 12
        assert tiles * 4 <= pieces < 2 ** 31 + 1000, (nx, ny, nz, pieces)
