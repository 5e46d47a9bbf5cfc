"""tsu_step_n_noalloc in FP64 on a grid so wide that even one chunk of rows has more tiles than its fixed
array has partial sums: the call reaches its launch (there is no device here: TSU_ECUDA) instead of looking for
a number of rows for ever.  The addresses point nowhere, so this runs where no GPU is visible."""
import os
import subprocess
import sys

from paper_2005_11931_gb300 import build

CODE = """
import sys; sys.path.insert(0, %r)
from paper_2005_11931_gb300 import tsu
g = tsu.Grid(8200000, 3, 8200000, 1 / 8199999, 0.5)
med = tsu.Medium(1 << 20, 1 << 20, 1.0, 1.0, 1.0, 1.0)
st = tsu.State()
st.buf[0], st.buf[1], st.nbuf, st.form, st.cur, st.aux = 1 << 20, 1 << 21, 2, tsu.TSU_FORM_STANDARD, 1, 0
try:
    tsu.tsu_step_n_noalloc(g, "f64", 1e-8, med, st, 1, energy=None, stream=0)
except tsu.TsuError as e:
    assert e.code == tsu.TSU_ECUDA, e
    print("PASS")
"""


def test_returns():
    build.build()
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    env = dict(os.environ, CUDA_VISIBLE_DEVICES="")
    r = subprocess.run([sys.executable, "-c", CODE % root], env=env, cwd=root, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and "PASS" in r.stdout, r.stdout + r.stderr
