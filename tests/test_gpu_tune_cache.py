"""A plan reads its autotune cache once, so that all its decisions rest on the same contents whatever happens to
the file meanwhile: here a named pipe, whose first reader gets the picks and every later one nothing."""
import os
import re
import threading
import time

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import oracle as O
from paper_1909_05600_gb300 import ffm, workloads as W

pytestmark = pytest.mark.gpu


def _tuned(X, kernel, u, path, pick, **kw):
    """Cache file of an autotuned plan with every Lagrange pick set to `pick`; the plan's own product."""
    with ffm.Plan(X, X, kernel, 0.0, 1e-3, **kw) as p:
        v = p.apply(u)
        p.autotune(cache_path=str(path))
    lines = [ln.split(" = ")[0] + " = %d" % pick if ln.startswith("lag ") else ln
             for ln in path.read_text().splitlines()]
    assert any(ln.startswith("lag ") for ln in lines)
    path.write_text("\n".join(lines) + "\n")
    return v.double()


def test_picks_belong_to_a_kernel_and_to_its_kernels_generation(tmp_path):
    X = torch.as_tensor(W.cube_volume(20000, 1), device="cuda")
    u = torch.ones(20000, device="cuda")
    path = tmp_path / "picks"
    _tuned(X, ffm.LAPLACE, u, path, 0, r1_override=4)
    lines = path.read_text()
    levels = lambda p: [p.info()["tune_tc"][l] for l in range(22) if p.info()["n_adm"][l]]
    with ffm.Plan(X, X, ffm.LAPLACE, 0.0, 1e-3, r1_override=4, autotune_cache=str(path)) as p:
        assert levels(p) and not any(levels(p))
    for kernel, kw in ((ffm.LAPLACE_GRAD, {}), (ffm.LAPLACE_DL, dict(normals=X))):
        with ffm.Plan(X, X, kernel, 0.0, 1e-3, r1_override=4, autotune_cache=str(path), **kw) as p:
            assert levels(p) and all(levels(p))
    # a pick timed on earlier kernels (keys without kind and generation)
    path.write_text(re.sub(r" gen=\d+ kind=\d+", "", lines))
    with ffm.Plan(X, X, ffm.LAPLACE, 0.0, 1e-3, r1_override=4, autotune_cache=str(path)) as p:
        assert all(levels(p))
    # complex levels have no pick, and build nothing for one
    path.write_text("".join(ln.replace("kind=0", "kind=1") + "\n" for ln in lines.splitlines() if ln.startswith("lag ")))
    size = []
    for cache in (None, str(path)):
        with ffm.Plan(X, X, ffm.HELMHOLTZ, 1.0, 1e-3, r1_override=4, kappa_switch=1e9, autotune_cache=cache) as p:
            size.append(p.bytes())
            assert all(levels(p))
    assert size[0] == size[1]


@pytest.mark.parametrize("pick", [0, 1, 2])
def test_the_cache_is_read_once(pick, tmp_path):
    X = torch.as_tensor(W.cube_volume(20000, 1), device="cuda")
    u = torch.as_tensor(np.random.default_rng(1).standard_normal(20000).astype(np.float32), device="cuda")
    v = _tuned(X, ffm.LAPLACE, u, tmp_path / "picks", pick)
    pipe, served, stop = tmp_path / "pipe", [], []
    os.mkfifo(pipe)

    def serve():
        while not stop:
            with open(pipe, "w") as f:  # until the next reader
                if not served:
                    f.write((tmp_path / "picks").read_text())
                served.append(1)
            time.sleep(0.3)  # until this reader has closed its end

    t = threading.Thread(target=serve, daemon=True)
    t.start()
    with ffm.Plan(X, X, ffm.LAPLACE, 0.0, 1e-3, autotune_cache=str(pipe)) as p:
        stop.append(1)
        reads = len(served)
        os.close(os.open(pipe, os.O_RDONLY | os.O_NONBLOCK))  # releases a writer that waits for a reader
        info = p.info()
        lag = [l for l in range(info["l_stop"] + 1) if info["n_adm"][l]]
        assert reads == 1 and lag and all(info["tune_tc"][l] == pick for l in lag)
        got = p.apply(u).double()
        assert p.info()["device_errors"] == 0
    assert float((got - v).norm() / v.norm()) < 3e-6
