"""The autotuner's cache file: choices written for other sets of schedules
(lines without the present set's fields) are tuned again, and a choice holds
for the row layout and the program it was timed with."""
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def M():
    import torch
    assert torch.cuda.is_available()
    import paper_2009_03052_gb300 as M
    M.build()
    M.load()
    yield M
    M.autotune(1, "")


def test_old_choices_are_tuned_again(M, tmp_path):
    g, k, bits = synth.grid_road(83, seed=1), 5, 64
    G = M.Graph.from_csr(g)
    key = G.info()
    b = M.autotune_choice  # (kind, k, bits, h, n, nnz, max degree) -> choice
    path = tmp_path / "tune.txt"
    import math
    n, nnz, maxd = key
    bucket = f"{int(math.log2(n))} {int(2 * math.log2(nnz / n))} {int(math.log2(maxd + 1))}"
    path.write_text("".join(f"{kind} {k} {bits} {h} {bucket} 5\n"
                            for kind in (0, 1) for h in range(2, k + 1 - (kind == 0))))
    old = path.read_text()
    M.autotune(1, str(path))
    assert b(1, k, bits, 3, *key) == 5
    M.Tables(G, synth.balanced_colors(g.n, k, 1), k, bits).free()
    new = path.read_text()
    assert new.startswith(old) and len(new.splitlines()) == len(old.splitlines()) + (k - 1) + (k - 2)
    # and the lines it wrote are not
    M.Tables(G, synth.balanced_colors(g.n, k, 2), k, bits).free()
    assert path.read_text() == new
    # a pinned choice is
    M.autotune_set(1, k, bits, 3, *key, 4)
    M.Tables(G, synth.balanced_colors(g.n, k, 2), k, bits).free()
    assert path.read_text() == new and b(1, k, bits, 3, *key) == 4


def test_programs_are_tuned_apart(M, tmp_path):
    # level k of a round-skipped build runs another merge program
    g, k, bits = synth.grid_road(91, seed=2), 6, 128
    G = M.Graph.from_csr(g)
    path = tmp_path / "tune.txt"
    M.autotune(1, str(path))
    colors = synth.balanced_colors(g.n, k, 1)
    M.Tables(G, colors, k, bits, skip_round=True).free()
    skip = path.read_text().splitlines()
    M.Tables(G, colors, k, bits).free()
    full = path.read_text().splitlines()[len(skip):]
    # level k - 1 (merge and sums) was not built before; level k's merge is another
    assert sorted(x.split()[0] + x.split()[3] for x in full) == sorted([f"1{k - 1}", f"0{k - 1}", f"1{k}"])
