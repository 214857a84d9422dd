"""The cuts of the acceptance kernel at their edges: vocabularies around the block's width, cuts that fall
among equal values, rows that do not spread over the kernel's bins."""
import numpy as np
import pytest
import torch

from oracle import ssd_oracle as orc
from paper_2505_15380_b200 import synth
from tests.gpu_case import _nucleus_edge_close

pytestmark = pytest.mark.gpu


def _rows(kind, n, V, rng):
    z = rng.standard_normal((n, V))
    if kind == "ties":          # many equal values: the cut falls among them
        z = np.round(z * 2) / 2 + 0.0  # (no negative zeros)
    elif kind == "flat":        # one value
        z[:] = 0.25
    elif kind == "outlier":     # one id far below: all others in one bin
        z[:, V // 2] = -1e6
    elif kind == "peaked":
        z *= 6.0
    return z.astype(np.float32)


@pytest.mark.parametrize("kind", ["normal", "ties", "flat", "outlier", "peaked"])
@pytest.mark.parametrize("V", [2, 33, 1024, 1025, 6564, 46080])
def test_cuts(V, kind):
    from paper_2505_15380_b200 import binding
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(V)
    B, gamma = 4, 2
    compared = 0
    for top_k, top_p, temperature in [(0, 0.0, 1.0), (1, 0.0, 0.7), (25, 0.0, 0.8), (0, 0.77, 1.0), (600, 0.77, 1.3),
                                      (V - 1, 0.03, 1.0)]:
        lg = _rows(kind, B * (gamma + 1), V, rng).reshape(B, gamma + 1, V)
        p = synth.random_prob_rows(B * gamma, V, seed=V, sharpness=1.0).reshape(B, gamma, V)
        x = synth.sample_from_rows(p.reshape(-1, V), seed=V + 1).reshape(B, gamma).astype(np.int32)
        u = synth.verify_uniforms(V, B, gamma + 1, step=top_k)
        k, y = (torch.full((B,), -2, dtype=torch.int32, device=dev) for _ in range(2))
        t = [torch.from_numpy(a).to(dev).contiguous() for a in (lg, x, p, u)]
        binding.accept_noalloc(*t, binding.VerifyParams(gamma, temperature, top_k, 0.2, top_p), k, y)
        torch.cuda.synchronize()
        for b in range(B):
            z = (lg[b] * np.float32(1.0 / temperature)).astype(np.float64)
            if any(_nucleus_edge_close(r, 1.0, top_k, top_p) for r in z):
                continue
            q = np.stack([orc.transform(r, 1.0, top_k, top_p) for r in z])
            o = orc.accept_step(q, p[b], x[b], u[b], 0.2)
            if any(abs(a - float(u[b, i, 0])) < 1e-3 for i, a in enumerate(o["thresholds"])):
                continue
            assert int(k[b]) == o["k"]
            if o["draw_margin"] >= 1e-5:
                assert int(y[b]) == o["y"]
                compared += 1
    assert compared >= 8


@pytest.mark.parametrize("B", [1, 19, 40])
@pytest.mark.parametrize("V", [2, 7, 1025, 2047, 6564, 46080])
def test_plain_rows(V, B):
    """Softmax over the whole vocabulary, on both sides of the number of rows up to which a cluster takes a row."""
    from paper_2505_15380_b200 import binding
    dev = torch.device("cuda:0")
    rng = np.random.default_rng(V + B)
    gamma = 4
    lg = _rows("normal", B * (gamma + 1), V, rng).reshape(B, gamma + 1, V)
    p = synth.random_prob_rows(B * gamma, V, seed=V, sharpness=1.0).reshape(B, gamma, V)
    x = synth.sample_from_rows(p.reshape(-1, V), seed=V + 1).reshape(B, gamma).astype(np.int32)
    u = synth.verify_uniforms(V, B, gamma + 1)
    k, y = (torch.full((B,), -2, dtype=torch.int32, device=dev) for _ in range(2))
    compared = 0
    for beta in (0.0, 0.4):
        t = [torch.from_numpy(a).to(dev).contiguous() for a in (lg, x, p, u)]
        binding.accept_noalloc(*t, binding.VerifyParams(gamma, 1.0, 0, beta), k, y)
        torch.cuda.synchronize()
        for b in range(B):
            q = np.stack([orc.transform(r.astype(np.float64), 1.0, 0) for r in lg[b]])
            o = orc.accept_step(q, p[b], x[b], u[b], beta)
            if any(abs(a - float(u[b, i, 0])) < 1e-5 for i, a in enumerate(o["thresholds"])):
                continue
            assert int(k[b]) == o["k"]
            if o["draw_margin"] >= 1e-5:
                assert int(y[b]) == o["y"]
                compared += 1
    assert compared >= B
