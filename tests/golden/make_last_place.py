"""Write tests/golden/last_place.txt on a GB300 (run from the repository root):
the digests of tests/test_gpu_last_place.py.  The committed file was written
with the library of commit 54c91b5, before its kernels were reorganised for
speed."""
import os
import sys

sys.path.append(os.getcwd())
import paper_2011_10658_gb300 as q   # noqa: E402
from tests import test_gpu_last_place as t   # noqa: E402

out = {}
for case in t.MOVES:
    out.update(t.move_digests(q, *case))
for case in t.PRODUCTS:
    out.update(t.product_digests(q, *case))
for case in t.UPDATES:
    out.update(t.update_digests(q, *case))
for node in (0, 32, 56):
    out.update(t.update_digests(q, (4, 4, 4), 32, "tf32x3", node, 64, t.ODD))
for k, v in out.items():
    print(k, v)
