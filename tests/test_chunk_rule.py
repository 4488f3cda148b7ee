"""How the sources of FP64 evaluations are split into chunks (chunk_rule.cuh), compiled for the host.

Even batches are split as the single network is.  In a batch with one large realisation among many
tiny ones neither the work list nor the partial forces may grow as n_r^2 / mean.
"""

import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2005_02498_gb300", "csrc")
SLOTS = 152 * 16
PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include "chunk_rule.cuh"
int main(int argc, char** argv)  // n <nodes> | len <tiles> <sources> | batch <longest> <targets> <n> <count> ...
{
    const long long slots = atoll(argv[1]);
    if (argv[2][0] == 'n') printf("%d\n", ptadd::network_max_chunks(atoll(argv[3])));
    if (argv[2][0] == 'l') printf("%lld\n", (long long)ptadd::chunk_len_rule(slots, atoll(argv[3]), atoll(argv[4])));
    if (argv[2][0] == 'b') {
        const long long targets = atoll(argv[4]);  // per realisation at most
        std::vector<int64_t> n;
        for (int i = 5; i + 1 < argc; i += 2) n.insert(n.end(), atoi(argv[i + 1]), atoll(argv[i]));
        long long tiles = 0, items = 0, bytes = 0;
        for (int64_t k : n) tiles += (std::min<long long>(k, targets) + 31) / 32;
        const std::vector<int64_t> len = ptadd::batch_chunk_lens(slots, tiles, n, atoll(argv[3]));
        for (size_t r = 0; r < n.size(); ++r) {
            const long long ch = (n[r] + len[r] - 1) / len[r];
            items += (std::min<long long>(n[r], targets) + 31) / 32 * ch;
            bytes += 48 * n[r] * ch;
        }
        printf("%lld %lld %lld %lld\n", (long long)len.front(), (long long)len.back(), items, bytes);
    }
}
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("chunk_rule")
    (d / "rule.cpp").write_text(PROGRAM)
    subprocess.run(["g++", "-O1", "-std=c++17", "-I" + CSRC, "-x", "c++", str(d / "rule.cpp"), "-o", str(d / "rule")], check=True)

    def run(*args):
        out = subprocess.run([str(d / "rule"), str(SLOTS), *map(str, args)], check=True, capture_output=True, text=True)
        return [int(v) for v in out.stdout.split()]
    return run


@pytest.mark.parametrize("R,n", [(1, 21), (9, 512), (16, 2000), (40, 4000), (2, 8192)])
def test_even_batches_follow_the_single_network(rule, R, n):
    """every realisation in the chunks that the rule gives for its size and all tiles"""
    tiles = R * ((n + 31) // 32)
    (fine,) = rule("len", tiles, n)
    first, last, items, _ = rule("batch", 2048, n, n, R)
    assert first == last == min(2048, fine) and items == tiles * -(-n // fine)


@pytest.mark.parametrize("sizes", [[(16384, 1), (200, 63)], [(50000, 1), (64, 255)], [(100000, 1), (2, 1000)],
                                   [(4000, 1), (5, 96)], [(1000000, 1), (100, 10000)]])
def test_one_large_realisation_among_many(rule, sizes):
    """At most four times the mean realisation's chunks: items <= 4 x tiles x those, and parts of the same order
    (these cases held 0.3, 2.3 and 14 GB at equal chunk lengths, the last one 480 GB)."""
    flat = [v for s in sizes for v in s]
    R, n = sum(c for _, c in sizes), sum(k * c for k, c in sizes)
    tiles = sum(c * ((k + 31) // 32) for k, c in sizes)
    (fine,) = rule("len", tiles, n // R)
    most = 4 * -(-(n // R) // fine)
    first, last, items, bytes_ = rule("batch", 10 ** 9, 10 ** 9, *flat)
    assert last == fine or last >= sizes[-1][0]
    assert -(-sizes[0][0] // first) <= most
    assert items <= most * tiles
    assert bytes_ <= 1 << 30


@pytest.mark.parametrize("sizes,targets,longest", [([(100000, 10)], 64, 2048), ([(200000, 3), (2, 5)], 32, 4096)])
def test_few_targets_among_many_sources(rule, sizes, targets, longest):
    """Parts over 1 GB only where the longest chunk allowed gives them."""
    flat = [v for s in sizes for v in s]
    *_, bytes_ = rule("batch", longest, targets, *flat)
    assert bytes_ <= max(1 << 30, sum(48 * k * c * -(-k // longest) for k, c in sizes))


@pytest.mark.parametrize("n,most", [(2, 512), (43690, 512), (43691, 511), (349525, 64), (1 << 30, 64)])
def test_chunks_of_a_single_network(rule, n, most):
    """512 while their parts stay below 1 GB, never fewer than 64"""
    assert rule("n", n) == [most]
