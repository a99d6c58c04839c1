"""The rules of the resident kernel that need no GPU (csrc/lbm_resident_rules.h), compiled here as
plain C++ and held against what the scheme does."""
import os
import random
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_1909_04166_gb300", "csrc")

EX = (0, 1, 0, -1, 0, 1, -1, -1, 1)
EY = (0, 0, 1, 0, -1, 1, 1, -1, -1)


def compiled(tmp_path, body, stdin=""):
    """Run a C++ program `body` that includes the rules; its output lines, split."""
    src, exe = tmp_path / "rules.cpp", tmp_path / "rules"
    src.write_text('#include <cstdio>\n#include "lbm_resident_rules.h"\nusing namespace cmlbm;\n'
                   + body)
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, "-o", str(exe), str(src)], check=True)
    out = subprocess.run([str(exe)], input=stdin, check=True, capture_output=True,
                         text=True).stdout
    return [line.split() for line in out.splitlines()]


def landings(row, width, sides, top=None, wall=0):
    """Words (row, column, plane) that the nodes of `row` push: population a lands at x + e_a;
    crossing a no-slip side (1) it comes back reversed to its node, crossing free-slip sides (2)
    alone it lands mirrored on this side of them; 0: no wall there.  top: the wall row, its kind."""
    index = {(x, y): a for a, (x, y) in enumerate(zip(EX, EY))}
    for c in range(width):
        for a in range(9):
            kx = sides[0] if c + EX[a] < 0 else sides[1] if c + EX[a] >= width else 0
            ky = wall if row == top and EY[a] > 0 else 0
            if 1 in (kx, ky) or (kx and ky):
                yield row, c, index[(-EX[a], -EY[a])]
            else:
                yield (row + (0 if ky else EY[a]), c + (0 if kx else EX[a]),
                       index[(-EX[a] if kx else EX[a], -EY[a] if ky else EY[a])])


@pytest.mark.parametrize("width", [1, 2, 37, 63, 64])
def test_carried_words_are_nobody_elses_and_complete(tmp_path, width):
    """The words that a round copies from the carry into its first row are those that the round
    before pushed there (beside words that a neighbouring block's message fills later), and none
    that the round itself pushes: the copy and the pushes have no barrier between them."""
    table = compiled(tmp_path, f"""
int main() {{
    for (int l = 0; l < 2; ++l) for (int r = 0; r < 2; ++r)
        for (int p = 2; p < 7; ++p) for (int c = -1; c <= {width}; ++c)
            if (p == 2 || p > 4) printf("%d %d %d %d %d\\n", l, r, p, c,
                                        (int)carry_fills(p, c, {width}, l, r));
}}""")
    copies = {}
    for l, r, p, c, on in (map(int, t) for t in table):
        copies.setdefault((l, r), set()).update({(c, p)} if on else set())
    first = 17
    for left in (0, 1, 2):
        for right in (0, 1, 2):
            for top, wall in ((None, 0), (first, 1), (first, 2), (first + 1, 1), (first + 1, 2)):
                sides, copied = (left, right), copies[left == 1, right == 1]
                before = {(c, a) for r, c, a in landings(first - 1, width, sides) if r == first}
                rows = [first] if top == first else [first, first + 1]
                during = {(c, a) for row in rows
                          for r, c, a in landings(row, width, sides, top, wall) if r == first}
                assert before <= copied
                assert not copied & during, (sides, top, wall)
                for c, a in copied - before:   # the rest: from beyond the strip, or a ghost node
                    assert not 0 <= c < width or not 0 <= c - EX[a] < width
                    assert not (c == 0 and left == 1 and a == 5)
                    assert not (c == width - 1 and right == 1 and a == 6)


PLAN = """
int main() {
    int nsm, fit, nx, ny;
    std::vector<GridSize> G;
    if (std::scanf("%d %d", &nsm, &fit) != 2) return 1;
    while (std::scanf("%d %d", &nx, &ny) == 2) G.push_back({nx, ny});
    for (const Wave& w : batch_waves(G, nsm, fit)) {
        for (const WavePart& p : w) std::printf("%d %d %d %d ", p.c, p.nstrip, p.nseg, p.h);
        std::printf("\\n");
    }
}"""


@pytest.mark.parametrize("n,lo,hi", [(1, 2, 3), (5, 2, 700), (30, 32, 256), (192, 32, 256),
                                     (300, 2, 64), (60, 300, 500)])
@pytest.mark.parametrize("fit", [32, 36])
def test_waves_hold_every_case_once_and_the_largest_comes_first(tmp_path, n, lo, hi, fit):
    """A launch that the device refuses has to be the first one of a run: the waves come in
    descending numbers of blocks."""
    rng = random.Random(n * fit + hi)
    grids = [(rng.randint(lo, hi), rng.randint(lo, hi)) for _ in range(n)]
    src = f"152 {fit}\n" + "\n".join(f"{x} {y}" for x, y in grids)
    waves = [[tuple(map(int, w[i:i + 4])) for i in range(0, len(w), 4)]
             for w in compiled(tmp_path, PLAN, src)]
    if any(-(-x // 64) * -(-y // fit) > 152 for x, y in grids):
        assert not waves
        return
    assert sorted(c for w in waves for c, *_ in w) == list(range(n))
    for w in waves:
        for c, nstrip, nseg, h in w:
            nx, ny = grids[c]
            assert nstrip == -(-nx // 64) and h == -(-ny // nseg) <= fit
            assert ny // nseg >= 2 or ny < 2
    blocks = [sum(nstrip * nseg for _, nstrip, nseg, _ in w) for w in waves]
    assert blocks == sorted(blocks, reverse=True) and blocks[0] <= 152


def test_a_plan_without_host_memory_is_no_plan(tmp_path):
    """Whichever allocation fails while a batch is planned, the plan is empty and nothing is thrown
    (the plan is made inside a C entry point)."""
    out = compiled(tmp_path, """
#include <cstdlib>
static int left = -1;
void* operator new(std::size_t n)
{
    if (left == 0) throw std::bad_alloc();
    if (left > 0) --left;
    return std::malloc(n);
}
void operator delete(void* p) noexcept { std::free(p); }
void operator delete(void* p, std::size_t) noexcept { std::free(p); }
int main()
{
    std::vector<GridSize> G;
    for (int i = 0; i < 40; ++i) G.push_back({40 + 5 * i, 250 - 3 * i});
    const size_t all = batch_waves(G, 152, 36).size();
    int failed = 0;
    for (int k = 0;; ++k) {
        left = k;
        const size_t n = batch_waves(G, 152, 36).size();
        const bool ran_out = left == 0;
        left = -1;
        if (!ran_out || n == all) break;
        if (n != 0) return 1;
        ++failed;
    }
    std::printf("%d %d\\n", failed, (int)all);
}""")
    failed, waves = map(int, out[0])
    assert failed > 20 and waves > 1
