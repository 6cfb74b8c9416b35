"""The anchor kernels at the lines of their dispatch (tiles of 32, 64 and 128
anchors, clusters of 8 and 2 blocks) against the FP64 oracle."""
import numpy as np
import pytest
import torch

from oracle import anchors as oa
from paper_2510_12174_gb300 import scenes
from paper_2510_12174_gb300.anchors import DeviceAnchors

pytestmark = pytest.mark.gpu

# on 152 SMs: 114 tiles of 32 anchors take clusters of 8; 19456 anchors the wider
# tiles (128 anchors, or 64 where the widest branches leave no room for 128)
CASES = [(3648, 3, 5), (3649, 3, 5), (19456, 4, 8), (19457, 16, 64)]


@pytest.fixture(scope="module", autouse=True)
def _built():
    import __graft_entry__ as ge
    ge.build()
    torch.cuda.set_device(0)


@pytest.mark.parametrize("A,M,C", CASES)
def test_decode_and_backward(A, M, C):
    """Outputs within 1e-5 of max(|ref|, 1).  Gradients by their norm: a
    parameter's is a float32 sum of A terms of order one and random sign, whose
    rounding is some 1e-6 of sqrt(A) however far the sum cancels."""
    arrs, mlps = scenes.anchor_set(A, M, C, seed=A + M)
    rng = np.random.default_rng(A)
    N = A * M
    up = {"mean": rng.normal(size=(3, N)), "quat": rng.normal(size=(4, N)),
          "scale": rng.normal(size=(3, N)), "opacity": rng.normal(size=N),
          "kfac": rng.normal(size=N), "sh": rng.normal(size=(N, 1, 3)),
          "sem": rng.normal(size=(N, C))}
    up = {k: v.astype(np.float32) for k, v in up.items()}
    da = DeviceAnchors.from_arrays(arrs, mlps)
    ds = da.decode()
    g = da.decode_backward({k: torch.as_tensor(v, device="cuda") for k, v in up.items()})
    torch.cuda.synchronize()
    ref = {k: v.detach().numpy() for k, v in oa.decode(oa.Anchors.from_arrays(arrs, mlps)).items()}
    for k, r in ref.items():
        got = getattr(ds, k).cpu().numpy().astype(np.float64).reshape(r.shape)
        assert (np.abs(got - r) / np.maximum(np.abs(r), 1.0)).max() < 1e-5, k
    rg, rm = oa.decode_and_grad(arrs, mlps, {k: v.astype(np.float64) for k, v in up.items()})[-2:]
    flat = {"pos": g["pos"].T, "scale": g["scale"].T}
    flat.update({k: g[k] for k in ("offsets", "feat", "sem", "kfac")})
    flat.update({f"{n}.{k}": v for n, d in g["mlps"].items() for k, v in d.items()})
    want = dict(rg)
    want.update({f"{n}.{k}": v for n, d in rm.items() for k, v in d.items()})
    for k, r in want.items():
        r = np.asarray(r, dtype=np.float64)
        d = np.linalg.norm(flat[k].cpu().numpy().astype(np.float64).reshape(r.shape) - r)
        assert d < 1e-5 * max(np.linalg.norm(r), np.sqrt(A)), (k, d, np.linalg.norm(r))
