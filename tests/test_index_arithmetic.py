"""The kernels' loop and launch arithmetic at the top of the ranges that the entry points accept, on the host: the helpers are
compiled from the kernel headers into a small program (no GPU is needed), and their walks are compared with Python's integers."""
import os
import subprocess

import pytest

from paper_2412_20386_b200 import build as lib_build
from test_gpu_short_k import RELOADS

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2412_20386_b200", "csrc")
INT_MAX = 2 ** 31 - 1

PROGRAM = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <vector>
#include "ptq_calibrate.cuh"
#include "ptq_gemm.cuh"
#include "ptq_quantize.cuh"
#include "ptq_short_k.cuh"

// quant images chunks_per_image sms: images between two of a thread, ring depth, images of one launch
static int quant(char **a)
{
    printf("%d %d %d\n", ptq::quant_image_step(atoi(a[0]), atoll(a[1]), atoi(a[2])), ptq::kQuantRingDepth, ptq::kQuantMaxImages);
    return 0;
}

// tiles elements: tiles visited, elements in them, start of the last one
static int tiles(char **a)
{
    long long visited = 0, elements = 0, last = -1;
    for (ptq::SearchTiles t(atoi(a[0])); t.valid() && visited < 4000000; t.next()) {
        ++visited;
        elements += t.count();
        last = t.at;
    }
    printf("%lld %lld %lld\n", visited, elements, last);
    return 0;
}

// shares Bc T sms: images of a block, blocks per position
static int shares(char **a)
{
    const ptq::CalibShares s = ptq::calib_shares(atoi(a[0]), atoi(a[1]), atoi(a[2]));
    printf("%d %d\n", s.images, s.blocks);
    return 0;
}

// plan elements T C sms: candidates per block, threads
static int plan(char **a)
{
    const ptq::SearchPlan p = ptq::search_plan(atoi(a[0]), atoi(a[1]), atoi(a[2]), atoi(a[3]));
    printf("%d %d\n", p.candidates, p.threads);
    return 0;
}

// units m_tiles n_tiles group sms k_blocks (group 0: as the few-channels kernel takes it): tiles visited other than once, most units of a CTA, most of a CTA's 24 per unit and 4 per change of
// its weights, 1 where CTAs keep to their groups, most loads of weights of a CTA
static int units(char **a)
{
    ptq::UnitParams p = {};
    p.m_tiles = atoi(a[0]);
    p.n_tiles = atoi(a[1]);
    p.group = atoi(a[2]) ? atoi(a[2]) : ptq::short_k_group(p.m_tiles, p.n_tiles, atoi(a[3]));
    p.groups = (p.n_tiles + p.group - 1) / p.group;
    p.N = 256 * p.n_tiles;
    p.k_blocks = atoi(a[4]);
    const long long total = (long long)p.m_tiles * p.groups;
    const int grid = (int)(total < atoi(a[3]) ? total : atoi(a[3]));
    ptq::set_units(p, grid);
    std::vector<int> visits((size_t)p.m_tiles * p.n_tiles, 0);
    int most = 0, cost = 0, reloads = 0;
    for (int cta = 0; cta < grid; ++cta) {
        int own = 0, loads = 0, held = -1;
        for (ptq::UnitCursor c(p, cta); c.valid(); ++own) {
            if (c.grp() != held) ++loads;
            held = c.grp();
            for (int n = c.size(); n > 0; --n, c.advance())
                if (c.m_tile() < p.m_tiles && c.n_tile() < p.n_tiles) ++visits[(size_t)c.m_tile() * p.n_tiles + c.n_tile()];
        }
        if (own > most) most = own;
        if (loads > reloads) reloads = loads;
        if (24 * own + 4 * (loads - 1) > cost) cost = 24 * own + 4 * (loads - 1);
    }
    long long wrong = 0;
    for (int v : visits) wrong += v != 1;
    printf("%lld %d %d %d %d\n", wrong, most, cost, p.spread > 0 ? 1 : 0, reloads);
    return 0;
}

int main(int argc, char **argv)
{
    if (argc > 1 && !strcmp(argv[1], "quant")) return quant(argv + 2);
    if (argc > 1 && !strcmp(argv[1], "tiles")) return tiles(argv + 2);
    if (argc > 1 && !strcmp(argv[1], "shares")) return shares(argv + 2);
    if (argc > 1 && !strcmp(argv[1], "plan")) return plan(argv + 2);
    if (argc > 1 && !strcmp(argv[1], "units")) return units(argv + 2);
    return 2;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("index")
    (d / "index.cu").write_text(PROGRAM)
    exe = str(d / "index")
    subprocess.run([lib_build.nvcc_path(), "-gencode", "arch=compute_100a,code=sm_100a", "-std=c++17", "-I", CSRC, "-o", exe,
                    str(d / "index.cu")], check=True, stdout=subprocess.PIPE, stderr=subprocess.STDOUT)

    def run(*args):
        out = subprocess.run([exe] + [str(a) for a in args], check=True, stdout=subprocess.PIPE, text=True).stdout
        return [int(v) for v in out.split()]
    return run


# one token position of 1 to 8 channels puts the most images between two of a thread
@pytest.mark.parametrize("B,chunks,sms", [(1, 1, 148), (9, 197 * 48, 148), (2147483000, 1, 148), (INT_MAX, 1, 148), (INT_MAX, 3, 132),
                                          (2 ** 30 + 1, 1, 160), (257, 2 ** 30, 148)])
def test_quantize_image_counters_stay_in_32_bits(program, B, chunks, sms):
    """Every thread's image index plus the loads it looks ahead (the index starts below the step and ends below the images plus one
    step) fits an int in each part of the batch, and a part's threads together visit every image."""
    most = program("quant", 1, 1, sms)[2]
    for first in range(0, B, most):
        images = min(most, B - first)
        step, depth, _ = program("quant", images, chunks, sms)
        assert 1 <= step <= images and images + depth * step <= INT_MAX
        assert step * chunks <= max(chunks, sms * 4 * 256)          # the launch has at most one wave of threads, or one image


@pytest.mark.parametrize("elements", [1, 2047, 2048, 2049, 2147481600, 2147481601, INT_MAX])
def test_search_tiles_cover_every_element(program, elements):
    starts = range(0, elements, 2048)
    assert program("tiles", elements) == [len(starts), elements, starts[-1]]


@pytest.mark.parametrize("Bc,T", [(1, 1), (8, 197), (9, 2), (700, 2), (2147483352, 1), (2147483353, 1), (2147483641, 1), (INT_MAX, 1),
                                  (INT_MAX, 40)])
def test_calibration_shares_cover_every_image(program, Bc, T):
    images, blocks = program("shares", Bc, T, 148)
    assert 1 <= blocks <= min(-(-2 * 148 // T), -(-Bc // 8))
    assert (blocks - 1) * images < Bc <= blocks * images


@pytest.mark.parametrize("elements,T,C,want", [
    (3072, 197, 8, [9, 256]), (3072, 197, 20, [9, 128]), (3072, 197, 54, [9, 64]), (3072, 197, 81, [27, 128]), (3072, 197, 100, [27, 64]),
    (384, 3136, 1, [9, 64]), (384, 3136, 28, [9, 64]), (384, 3136, 81, [27, 64]), (24576, 49, 81, [9, 256]), (96, 197, 1, [9, 128]),
    (1, 1, 1, [9, 64]), (INT_MAX, 1, 4096, [9, 128]), (INT_MAX, 1048576, 4096, [27, 64])])
def test_search_blocks_fill_the_chip_and_no_more(program, elements, T, C, want):
    assert program("plan", elements, T, C, 148) == want


# row tiles, N tiles, N tiles per unit: groups that divide the CTAs and do not, left-over row tiles with few and with many changes of the
# weights, fewer units than CTAs, more groups than CTAs, last groups that are smaller
@pytest.mark.parametrize("m,n,group", [(1, 1, 1), (148, 7, 1), (190, 7, 1), (253, 7, 1), (37, 12, 1), (37, 11, 1), (59, 5, 1), (148, 5, 1), (394, 3, 1),
                                       (147, 6, 1), (113, 13, 1), (105, 2, 2), (1568, 2, 2), (100, 5, 2), (85, 8, 3), (291, 10, 2), (2, 235, 1),
                                       (3, 149, 1), (1, 400, 3), (200000, 7, 1)])
@pytest.mark.parametrize("sms", [148, 132])
def test_unit_order_visits_every_tile_once(program, m, n, group, sms):
    """No CTA has more units than an even split gives the busiest, and where there are CTAs enough for one group each, changes of the
    weights make no left-over CTA the one that the launch waits for by more than a twenty-fifth."""
    units = m * -(-n // group)
    rounds = -(-units // min(units, sms))
    groups = -(-n // group)
    for k_blocks in (1, 3):
        wrong, most, cost, spread, _ = program("units", m, n, group, sms, k_blocks)
        assert wrong == 0 and most == rounds
        if groups <= min(units, sms) and k_blocks > 1:
            assert cost <= max(25 * rounds, 24 * rounds + 4)
        if groups == 1:
            assert spread == 1
        if (m, n, group, sms) in ((148, 7, 1, 148), (37, 12, 1, 148)):
            assert spread == 0


def test_few_channel_layers_reload_their_weights(program):
    """The layers that the few-channels kernel is tested with for a change of weights within a CTA have one."""
    for K, N, T, M, bias, off in RELOADS:
        wrong, _, _, spread, loads = program("units", -(-M // 128), -(-N // 256), 0, 148, 1)
        assert wrong == 0 and loads > 1
