"""Table builds whose blocks hold nearly 48 KB of columns: static and dynamic shared
memory together pass the default limit there.  Each width is the first build of a
process (a wider one before it would have raised the limit), and the tables equal
those of the same materials built one at a time."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CODE = """
import sys
import numpy as np
from paper_1907_02814_gb300 import pcc
n, cols = int(sys.argv[1]), int(sys.argv[2])
ctx = pcc.Context(0)
mats = [pcc.material(79, 5.0 + z, 5.9e28, 300.0) for z in range(n)]
spec = pcc.table_spec(n_rows=5, n_cols=cols, quad_nodes=4)
ctx.tables_build(mats, spec)
t = ctx.tables_read()
for m in (0, n - 1):
    ctx.tables_build(mats[m:m + 1], spec)
    one = ctx.tables_read()
    for k in ("brems_sigma", "brems_cdf", "bh_sigma", "bh_cdf"):
        np.testing.assert_allclose(t[k][m], one[k][0], rtol=1e-12)
    assert np.all(t["brems_sigma"][m] > 0) and np.all(t["brems_cdf"][m][:, -1] == 1.0)
print("built")
"""


@pytest.mark.parametrize("n,cols", [(8, 730), (31, 742), (2, 3000), (4, 1500), (1, 4096)])
def test_widths_at_the_default_limit(n, cols):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1907_02814_gb300 import build
    build.build()
    r = subprocess.run([sys.executable, "-c", CODE, str(n), str(cols)], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0 and "built" in r.stdout, r.stderr[-2000:]
