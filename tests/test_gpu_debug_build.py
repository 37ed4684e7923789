"""The -DMONA_DEBUG build (libmona_debug.so): the kernels check their own indices - tile coordinates, slab positions,
staging offsets, the addresses of the axpy operand and of the parameters, slab ranges of the elementwise passes - and latch MONA_ERR_BOUNDS
in the status word instead of trapping.  It stands in for a memory checker where none is available.  The parity cases
with ragged tiles, padded batches, tall / wide / tiny shapes and both state formats run under it in a child process
(the library is chosen when the binding first loads it) and must come back clean and within tolerance."""
import os
import subprocess
import sys

import pytest

from paper_2605_26842_b200 import build as build_mod

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r"""
import torch
import paper_2605_26842_b200 as pkg
from paper_2605_26842_b200 import binding
from paper_2605_26842_b200.binding import FORM_FEW_TILES, FORM_MANY_TILES, FORM_WHOLE_MATRICES
from tests.parity_util import TOL_O_BF16, TOL_STATE, TOL_W, run_case
assert binding._LIB_PATH.endswith("libmona_debug.so"), binding._LIB_PATH
cases = [dict(shapes=[(1, 72, 200), (1, 1000, 136), (3, 192, 320), (2, 320, 192)], steps=2, seed=3),
         dict(shapes=[(5, 256, 768), (2, 768, 256), (1, 1024, 1536), (1, 32, 512), (1, 33, 17)], steps=2, seed=4),
         dict(shapes=[(3, 128, 384)], steps=3, seed=9, grad_dtype=torch.bfloat16, pad=64),
         dict(shapes=[(2, 512, 256), (1, 264, 520)], steps=3, seed=21, lite=True),
         dict(shapes=[(2, 2048, 768), (1, 1536, 2048)], steps=1, seed=5),
         dict(shapes=[(4, 256, 512)], steps=2, seed=6, options=pkg.default_options(fuse_update=1, ns_delay=1, macro_tile_min_k=64))]
# O is not asked for: the last product updates the parameters, in every form of the launch, with plain, narrow and wide tiles cut in both
# directions; whole matrices with A, B', C and the diagonal correction owned by a pair's lanes, or by the matrix
plain = [([(100, 520, 648)], FORM_MANY_TILES, 256, {}), ([(100, 648, 520)], FORM_MANY_TILES, 256, dict(pad=64)), ([(20, 520, 648)], FORM_MANY_TILES, 512, {}),
         ([(1, 264, 776)], FORM_FEW_TILES, 128, {}), ([(10, 1032, 1000)], FORM_FEW_TILES, 512, {}), ([(148, 248, 1016)], FORM_WHOLE_MATRICES, None, {}),
         ([(100, 200, 72)], FORM_WHOLE_MATRICES, 256, dict(pad=8)), ([(370, 712, 136)], FORM_WHOLE_MATRICES, None, dict(hp=pkg.default_hparams(ns_steps=7)))]
for shapes, form, columns, kw in plain:
    last = binding.describe_step([pkg.MatrixDesc(r, c, b, r * c + kw.get("pad", 0), 0, 0) for b, r, c in shapes], kw.get("hp"))[-1]
    assert last.form == form and last.update_columns > 0 and columns in (None, last.update_columns), (shapes, last.form, last.update_columns)
    cases.append(dict(kw, shapes=shapes, steps=1, seed=7, want_o=False, sample={0: sorted({0, shapes[0][0] // 2, shapes[0][0] - 1})}))
for kw in cases:
    errs = run_case(**kw)       # run_case polls the status word after every step and fails on anything but MONA_OK
    assert errs["M"] <= (3e-4 if kw.get("lite") else TOL_STATE), errs
    assert errs["O"] <= TOL_O_BF16 and errs["dW"] <= TOL_W, errs
print("debug build clean")
"""


@pytest.mark.gpu
def test_parity_cases_run_clean_under_the_index_checking_build():
    lib = build_mod.build(debug=True)
    env = dict(os.environ, MONA_LIBRARY=lib, PYTHONPATH=ROOT + os.pathsep + os.environ.get("PYTHONPATH", ""))
    res = subprocess.run([sys.executable, "-c", CHILD], cwd=ROOT, env=env, capture_output=True, text=True, timeout=900)
    assert res.returncode == 0, res.stdout[-2000:] + res.stderr[-4000:]
    assert "debug build clean" in res.stdout


def test_debug_build_exports_the_same_entry_points():
    import ctypes as C
    import re
    lib = C.CDLL(build_mod.build(debug=True))
    text = open(os.path.join(ROOT, "include", "mona.h")).read()
    text = re.sub(r"/\*.*?\*/", "", text, flags=re.S)
    for name in sorted(set(re.findall(r"\b(mona_[a-z_0-9]+)\s*\(", text))):
        assert hasattr(lib, name), name
