"""First calls of a process at sizes whose dynamic shared memory alone stays
below 48 KB and passes it with the kernel's static part: the opt-in must not
depend on a larger size having run before, so every case has a process of its
own.  The FP32 QR of the mixed path (panels of 32 columns at M = 81 and 93, of
16 at M = 179, tried by the autotuner) with its Q panels, the comb of 4096
walkers and the pair branching of 2048."""
import os
import subprocess
import sys

import pytest

pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

HEAD = """
import numpy as np, torch
import __graft_entry__
__graft_entry__.build()
import paper_2012_12228_gb300 as ftq
from synthetic_inputs import gaussian_fields
"""

# G against the complex128 path with the bound of the other mixed tests
QR = HEAD + """
M, N, tune = {M}, 14, {tune}
out = []
for precision in (ftq.FTQ_MIXED, ftq.FTQ_FP64):
    p = ftq.Propagator(N, M, 1.0, 0.25, 0.05, walkers=2, precision=precision)
    if tune and precision == ftq.FTQ_MIXED:
        p.autotune()
    p.propagate(torch.from_numpy(gaussian_fields(3, 6, 2, p.n_alpha)).cuda())
    assert p.status() == 0
    out.append(p.green().cpu().numpy())
assert np.abs(out[0] - out[1]).max() < 1e-5 * np.abs(out[1]).max()
"""

POPULATION = HEAD + """
from oracle.population import comb_counts, comb_pairs, pair_branch_pairs
W, comb = {W}, {comb}
p = ftq.Propagator(2, 7, 1.0, 0.5, 0.05, walkers=W)
p.propagate(3.0 * torch.from_numpy(gaussian_fields(5, 8, W, p.n_alpha)).cuda())
ws = p.weights().cpu().numpy()
lw = np.where(ws[:, 2] > 0.5, ws[:, 0], -np.inf)
w = np.exp(lw - lw.max())
if comb:
    pairs = comb_pairs(comb_counts(w, 0.37))
    parent = p.population_control(0.37)
else:
    draws = np.random.default_rng(7).random(W // 2)
    pairs = [(s, d) for s, d, _ in pair_branch_pairs(w, draws)]
    parent = p.pair_branch(draws)
assert pairs
ref = np.arange(W)
for s, d in pairs:
    ref[d] = s
assert np.array_equal(parent.cpu().numpy(), ref)
"""


@pytest.mark.parametrize("script", [
    pytest.param(QR.format(M=81, tune=False), id="qr81"), pytest.param(QR.format(M=93, tune=True), id="qr93"),
    pytest.param(QR.format(M=179, tune=True), id="qr179"),
    pytest.param(POPULATION.format(W=4096, comb=True), id="comb4096"),
    pytest.param(POPULATION.format(W=2048, comb=False), id="branch2048")])
def test_first_call_of_a_process(script):
    r = subprocess.run([sys.executable, "-c", script], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
