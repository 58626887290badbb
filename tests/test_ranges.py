"""Index arithmetic of the kernels (csrc/ranges.h), compiled for the host: what is touched, and that nothing else is."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2605_29986_b200", "csrc")


@pytest.fixture(scope="module")
def run_cpp(tmp_path_factory):
    folder = tmp_path_factory.mktemp("ranges")

    def run(name, body):
        src = folder / (name + ".cpp")
        src.write_text('#include "ranges.h"\n#include <cstdio>\n#include <cstdlib>\n#include <vector>\nusing namespace cfgzip;\n' + body)
        exe = str(folder / name)
        subprocess.check_call([shutil.which("g++") or "c++", "-O2", "-std=c++17", "-Wall", "-Werror", "-ftrapv", "-I", CSRC, "-o", exe, str(src)])
        out = subprocess.run([exe], stdout=subprocess.PIPE, text=True)
        assert out.returncode == 0, out.stdout
    return run


def test_every_piece_of_every_row_is_dealt_once(run_cpp):
    run_cpp("pieces", r"""
int main() {
    for (int B : {1, 2, 7, 100})
        for (int chunks : {1, 2, 3, 16, 63})
            for (unsigned blocks : {1u, 2u, 5u, 63u, 64u, 700u}) {
                std::vector<int> seen(size_t(B) * chunks, 0);
                for (unsigned b = 0; b < blocks; ++b)
                    for (PieceWalk at(b, chunks, int(blocks) / chunks, int(blocks) % chunks); at.row < B; at.next()) {
                        if (at.row < 0 || at.ch < 0 || at.ch >= chunks) { printf("B %d chunks %d: row %lld piece %d\n", B, chunks, (long long)at.row, at.ch); return 1; }
                        ++seen[size_t(at.row) * chunks + at.ch];
                    }
                for (int n : seen) if (n != 1) { printf("B %d chunks %d blocks %u: a piece %d times\n", B, chunks, blocks, n); return 1; }
            }
}
""")


def test_pieces_beyond_2_to_the_31(run_cpp):
    # the walk of the last blocks of a full grid ends behind the last row (32-bit counting of the pieces came round to the
    # front: 2^31 - 1 rows of one piece, or fewer of several)
    run_cpp("many", r"""
int main() {
    const unsigned blocks = 148 * 64;
    const int shapes[][2] = {{2147483647, 1}, {2147483647, 2}, {1500000000, 3}};
    for (auto& s : shapes)
        for (unsigned b : {0u, 1u, blocks - 1}) {
            long long last = -1, n = 0;
            for (PieceWalk at(b, s[1], int(blocks) / s[1], int(blocks) % s[1]); at.row < s[0]; at.next(), ++n) {
                const long long piece = (long long)at.row * s[1] + at.ch;
                if (at.row < 0 || at.ch < 0 || at.ch >= s[1] || piece != (long long)b + n * blocks || piece <= last) { printf("piece %lld after %lld\n", piece, last); return 1; }
                last = piece;
            }
            const long long total = (long long)s[0] * s[1];
            if (n != (total - b + blocks - 1) / blocks) { printf("%lld pieces for block %u\n", n, b); return 1; }
        }
}
""")


def test_octets_of_a_row_ask_for_its_tokens_and_nothing_else(run_cpp):
    # rows whose vectors start up to seven tokens in front of them (wherever the row starts in memory), every length around a
    # vector or two: a vector at either end that reaches past the row is read token by token
    run_cpp("octets", r"""
int main() {
    for (int V = 1; V <= 41; ++V)
        for (int lead = 0; lead < 8; ++lead) {
            std::vector<int> seen(size_t(V), 0);
            for (int t0 = -lead - 16; t0 <= V + 16; t0 += 8) {
                auto read = [&](int t) { if (t < 0 || t >= V) { printf("V %d lead %d: token %d\n", V, lead, t); exit(1); } ++seen[size_t(t)]; };
                octet_loads(t0, V, [&] { for (int q = 0; q < 8; ++q) read(t0 + q); },
                            [&] { for (int q = 0; q < 8; ++q) if (octet_has(t0, q, V)) read(t0 + q); });
            }
            for (int n : seen) if (n != 1) { printf("V %d lead %d: a token %d times\n", V, lead, n); return 1; }
        }
}
""")
