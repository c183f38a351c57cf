"""The rules that choose a call's kernel by its sizes (csrc/routes.h), against
measured times of both sides (tests/golden/*_routes.txt): the choice may not be
slower than the best by more than the times repeat, nor than the code that the
choice replaced."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2306_04235_gb300", "csrc")
GOLDEN = os.path.join(ROOT, "tests", "golden")

pytestmark = pytest.mark.skipif(shutil.which("g++") is None, reason="needs a host compiler")


def _decide(tmp_path, expr, rows):
    """The values of the C++ expression `expr` of ints a[] for every row."""
    src = tmp_path / "r.cpp"
    src.write_text(f"""#include "routes.h"
#include <cstdio>
using namespace mnmt;
int main() {{
    int n, a[16];
    while (scanf("%d", &n) == 1) {{
        for (int i = 0; i < n; i++) if (scanf("%d", a + i) != 1) return 1;
        printf("%d\\n", (int)({expr}));
    }}
}}
""")
    exe = tmp_path / "r"
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    text = "\n".join(f"{len(r)} " + " ".join(str(int(x)) for x in r) for r in rows)
    out = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True).stdout
    return [int(x) for x in out.split()]


def _table(name, kind):
    for line in open(os.path.join(GOLDEN, name)):
        f = line.split()
        if f and f[0] == kind:
            yield f[1:]


@pytest.mark.parametrize("kind", ["enc", "dec"])
def test_session_linears_take_the_faster_family(kind, tmp_path):
    rows = [([int(x) for x in f[:3]], float(f[3]), [float(x) for x in f[4:]]) for f in _table("linear_routes.txt", kind)]
    assert len(rows) > 60
    roles = "LIN_LAYER, LIN_SQUARE, LIN_CACHE".split(", ")
    got = [_decide(tmp_path, f"route_linear_tc({r}, a[0], a[1], a[2], a[1], a[1], false)", [x[0] for x in rows]) for r in roles]
    for (m, start, t), layer, square, cache in zip(rows, *got):
        column = 0 if not cache and not layer else 1 if not layer else 2 if not square else 3
        assert cache or not layer
        best = min(t)
        assert t[column] <= 1.06 * best, (m, t, column)
        assert not start or t[column] <= 1.01 * start + 2, (m, start, t, column)


def test_vocabulary_projection_takes_the_faster_family(tmp_path):
    rows = [([int(x) for x in f[:4]], float(f[4]), float(f[5])) for f in _table("linear_routes.txt", "out")]
    got = _decide(tmp_path, "route_linear_tc(LIN_OUT, a[0], a[2], 4 * a[2], a[1], a[2], a[3])", [x[0] for x in rows])
    for (m, t8, tc), choice in zip(rows, got):
        assert (tc if choice else t8) <= 1.06 * min(t8, tc), (m, t8, tc, choice)


# clusters of n CTAs that are resident at once on 152 SMs
FIT = {1: 152, 2: 76, 3: 45, 4: 36, 6: 23, 8: 15}


def test_batched_step_runs_where_it_is_faster(tmp_path):
    rows = [([int(x) for x in f[:4]], *map(float, f[4:])) for f in _table("rows_routes.txt", "rows")]
    assert len(rows) > 100
    taken = [0] * len(rows)
    for nb, hpc in ((1, 1), (2, 1), (4, 1), (2, 2)):
        args = [(beam, -(-r // (8 * nb)), FIT.get(heads // hpc, 0)) for (r, heads, beam, _), *_ in rows]
        for i, ok in enumerate(_decide(tmp_path, f"route_rows_variant({nb}, {hpc}, a[0], a[1], a[2])", args)):
            taken[i] |= ok
    for (m, batched, per_op, start), use in zip(rows, taken):
        t = batched if use else per_op
        # (one line for short and long sources: two beams cross between them)
        assert t <= 1.10 * min(batched, per_op), (m, batched, per_op, use)
        assert t <= 1.01 * start, (m, t, start)


def test_tcgen05_tiles_are_the_faster_ones(tmp_path):
    rows = [([int(x) for x in f[:4]], float(f[4]), [float(x) for x in f[5:]]) for f in _table("tc_routes.txt", "tc")]
    assert len(rows) > 300
    args = [(m, n, -(-k // 64), mode == 2, mode == 4, mode != 0 or n % 16 == 0) for (m, n, k, mode), *_ in rows]
    got = _decide(tmp_path, "route_tc_tiles(a[0], a[1], a[2], a[3], a[4], a[5], 152, 76)", args)
    loss = []
    for (m, start, t), choice in zip(rows, got):
        assert t[choice] <= 1.05 * start + 0.3, (m, start, t, choice)
        loss.append(t[choice] / min(t))
    assert sum(loss) / len(loss) < 1.03


def test_fake_quant_threads_are_not_idle(tmp_path):
    """Single elements get a thread each up to 8 blocks per SM; groups only where
    every array is aligned and they fill the blocks that single elements would."""
    sizes = [1, 100, 4095, 4096, 10007, 32767, 32768, 65536, 262143, 262144, 1 << 22]
    rows = [(n, al, bw, mm) for n in sizes for al in (0, 1) for bw in (0, 1) for mm in (0, 1)]
    call = "route_fake_quant(a[0], a[1], a[2], a[3], 152)"
    groups, blocks = _decide(tmp_path, call + ".groups", rows), _decide(tmp_path, call + ".blocks", rows)
    for (n, al, bw, mm), g, b in zip(rows, groups, blocks):
        per = (8 if bw else 4) if g else 1
        assert b == max(1, min(8 * 152, -(-(n // per) // 256)))
        assert not g or al
        if al:
            assert g == (n >= (262144 if bw and mm else 4096 if bw else 32768))


def test_layernorm_takes_the_faster_kernel(tmp_path):
    rows = [([int(x) for x in f[:2]], float(f[3]), float(f[4])) for f in _table("ln_routes.txt", "ln")]
    assert len(rows) > 100
    for (m, block, warp), choice in zip(rows, _decide(tmp_path, "route_layernorm_warp(a[0], a[1])", [x[0] for x in rows])):
        assert (warp if choice else block) <= 1.06 * min(block, warp), (m, block, warp, choice)
