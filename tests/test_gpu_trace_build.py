"""The -DMONA_TRACE build (libmona_trace.so): the Newton-Schulz kernel accounts for the cycles its roles wait and for the
MMA issuer's cycles and k-slices per kind of tile.  The instrumented kernel must compute what the ordinary one computes
(a parity case runs under it), and the counts it reports are exact, so they are checked against the tiling by hand:
k-slices per kind of tile, work items, CTAs.  The ordinary build must refuse the read-back instead of returning zeros."""
import json
import os
import subprocess
import sys

import pytest

from paper_2605_26842_b200 import build as build_mod

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import json, torch
import paper_2605_26842_b200 as pkg
from paper_2605_26842_b200 import binding
from tests.parity_util import TOL_O_BF16, TOL_STATE, TOL_W, run_case
assert binding._LIB_PATH.endswith("libmona_trace.so"), binding._LIB_PATH
errs = run_case(shapes=[(5, 256, 768), (2, 768, 256), (1, 1024, 1536)], steps=2, seed=4)
assert errs["M"] <= TOL_STATE and errs["O"] <= TOL_O_BF16 and errs["dW"] <= TOL_W, errs
binding.trace_read(reset=True, rows=0)
# 7 and 60 matrices 768 x 2048 (3 x 3 tile rows/columns of the small side, 8 tile columns of X), one step, 5 iterations
dev = torch.device("cuda", 0)
for mats in (7, 60):
    W = (torch.randn(mats, 768, 2048, device=dev) * 0.02)
    G = torch.randn(mats, 768, 2048, device=dev) * 1e-3
    opt = pkg.MonaOptimizer([W])
    last = binding.describe_step(opt.descs)[-1]
    opt.step(pkg.default_hparams(), [W], [G])
    torch.cuda.synchronize()
    assert opt.poll_status()[0] == 0
    rows = binding.trace_read(reset=True)
    again = binding.trace_read(reset=False)
    print("TRACE " + json.dumps({"mats": mats, "form": last.form, "update_columns": last.update_columns, "rows": rows, "again_sum": sum(map(sum, again))}))
    opt.close()
"""


@pytest.mark.gpu
def test_profiling_build_matches_the_oracle_and_counts_exactly():
    lib = build_mod.build(trace=True)
    env = dict(os.environ, MONA_LIBRARY=lib, PYTHONPATH=ROOT + os.pathsep + os.environ.get("PYTHONPATH", ""))
    res = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env, capture_output=True, text=True, timeout=900)
    assert res.returncode == 0, res.stdout[-2000:] + res.stderr[-4000:]
    runs = [json.loads(ln[len("TRACE "):]) for ln in res.stdout.splitlines() if ln.startswith("TRACE ")]
    assert [(d["mats"], d["form"], d["update_columns"]) for d in runs] == [(7, 1, 512), (60, 0, 256)]     # few tiles; many, the last product in plain tiles
    for d in runs:
        check_counts(d)


def check_counts(d):
    rows = [r for r in d["rows"] if r[0] > 0]
    assert d["again_sum"] == 0                      # the reset cleared the table
    assert len(rows) % 2 == 0 and 2 <= len(rows) <= 148
    lead = rows[0::2]
    mats = d["mats"]
    last_tiles = 12 if d["update_columns"] == 512 else 24          # work items of the product that updates the parameters
    # 768 x 768 symmetric products: 3 diagonal + 3 off-diagonal tiles; X X^T has 2048 / 64 = 32 k-slices, products of 768 x 768
    # matrices have 768 / 64 = 12; X' = B' X: 3 tile rows x 4 macro-tiles of 512 columns, 12 k-slices each.  768 x 2048 takes its
    # first two iterations together: one X X^T, P, P A, P (P A), P', P' P and one Q X; of the s x s products only P and P' have the
    # same operand on both sides, so the diagonal tiles of the other three count with the off-diagonal ones.  Three plain
    # iterations follow.
    macro, plain = (4, 0) if last_tiles == 12 else (3, 24)
    expect = {0: 4 * 3 * 32, 1: 4 * 3 * 32, 2: (5 + 3) * 3 * 12 + 3 * 3 * 12, 3: (2 + 3) * 3 * 12, 4: macro * 12 * 12, 5: plain * 12}
    for kind, per_matrix in expect.items():
        got = sum(r[16 + 4 * kind + 1] for r in lead)
        assert got == per_matrix * mats, (kind, got)
    assert sum(r[15] for r in rows) == 2 * ((6 * 6 + 12) + 2 * (6 + 6 + 12) + (6 + 6 + last_tiles)) * mats       # every item is counted once by each CTA of its pair
    for r in lead:
        for kind in range(5):
            cyc, ks, wf, wa = r[16 + 4 * kind:16 + 4 * kind + 4]
            assert wf + wa <= cyc
            # the tensor pipe needs 512 cycles per 256 x 256 x 64 step, twice that for a macro-tile
            # (the issuer runs a few k-slices ahead of the pipe, so a kind's average may dip a little below it)
            assert ks == 0 or cyc / ks >= (1024 if kind == 4 else 512) * 0.8, (kind, cyc, ks)
        assert r[4] <= r[5] and r[6] + r[7] <= r[8]          # a role's waits fit inside the role
    for r in rows:
        assert r[1] + r[2] <= r[3] and r[13] <= r[14] and r[9] + r[10] + r[11] <= r[12]


def test_ordinary_build_refuses_the_profiling_read_back():
    import paper_2605_26842_b200 as pkg
    from paper_2605_26842_b200 import binding
    if os.environ.get("MONA_LIBRARY"):
        pytest.skip("another build of the library was selected for this run")
    with pytest.raises(pkg.MonaError) as e:
        binding.trace_read()
    assert e.value.status == 10


def test_profiling_build_exports_the_same_entry_points():
    import ctypes as C
    import re
    lib = C.CDLL(build_mod.build(trace=True))
    text = open(os.path.join(ROOT, "include", "mona.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    for name in sorted(set(re.findall(r"\b(mona_[a-z_0-9]+)\s*\(", text))):
        assert hasattr(lib, name), name
