"""A driver without the tensor-map encoder: the CUDA-core handles and the
allocation-free call take kernels that do not need it; the others say so."""

import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CODE = """
import numpy as np, torch, oracle
from paper_1102_0148_gb300 import corr, synth

def err(V, R, N):
    A = np.abs(R[[oracle.baseline_index(i, i, N) for i in range(N)]])
    ii, jj = np.triu_indices(N)
    return np.max(np.abs(V - R) / np.sqrt(A[ii] * A[jj]))

N, S = 3, 65
for K in (16, 64, 256, 512, 1024, 2048, 4096):
    p, _ = synth.make_samples(N, S * K, K, seed=K)
    R, _ = oracle.correlate(p, N, K)
    x = torch.from_numpy(p.reshape(-1)).cuda()
    torch.cuda.synchronize()
    with corr.Correlator(N, K, "fp32_simt") as c:
        c.push(x, S * K)
        V, n = c.dump(fp64=True)
        assert n == S and err(V, R, N) <= 1e-5, K
        Y = torch.empty((N, S, K // 2), dtype=torch.complex64, device="cuda")
        corr.corr_debug_spectra(c.h, x.data_ptr(), S * K, Y.data_ptr())
    vis = torch.empty((N * (N + 1) // 2, K // 2), dtype=torch.complex64, device="cuda")
    corr.corr_correlate_noalloc(x, S * K, N, K, vis, torch.cuda.current_stream())
    assert err(vis.cpu().numpy(), R, N) <= 1e-5, K
for dt in ("fp32", "fp16", "fp8"):
    try:
        corr.corr_create(3, 64, dt)
    except corr.CorrError as e:
        assert e.code == corr.CORR_ECUDA, e
    else:
        raise SystemExit(dt + " handle without tensor maps")
print("ok")
"""


def test_without_the_encoder(lib):
    pytest.importorskip("torch")
    env = dict(os.environ, CORR_TEST_NO_TENSOR_MAPS="1", PYTHONPATH=ROOT)
    r = subprocess.run([sys.executable, "-c", CODE], cwd=ROOT, env=env, capture_output=True, text=True, timeout=120)
    assert r.returncode == 0 and r.stdout.strip().endswith("ok"), r.stdout + r.stderr
