"""Host side of the binding and of the autotuner, with fakes in place of the device."""
import types

import pytest

pytest.importorskip("torch")


@pytest.fixture(scope="module")
def tri():
    from paper_1609_01490_gb300 import build
    build.build()
    from paper_1609_01490_gb300 import tri as t
    return t


def test_stream_without_the_raw_handle(tri, monkeypatch):
    # a torch without the private function: the public current stream
    import torch
    monkeypatch.setattr(tri, "_raw_stream", None)
    monkeypatch.setattr(torch.cuda, "current_stream", lambda: types.SimpleNamespace(cuda_stream=1234))
    assert tri._stream(None) == 1234
    assert tri._stream(7) == 7 and tri._stream(types.SimpleNamespace(cuda_stream=9)) == 9


def test_autotuner_times_the_tiles_it_names(tri, monkeypatch):
    # every candidate runs at its own rho: 4 x 4 pairs per thread, exactly the Life tile
    from paper_1609_01490_gb300 import autotune
    calls = []
    for name in ("tri_edm", "tri_ca_step", "tri_ca_step_tile", "tet_at_energy"):
        monkeypatch.setattr(tri, name, lambda *a, _n=name, **k: calls.append((_n, a, k)))
    work = object.__new__(autotune._Workload)
    work.x = work.out = work.a = work.b = work.p = work.e = work.ws = None
    work.n, work.d = 6400, 3
    for kernel in autotune.KERNELS:
        work.kernel = kernel
        for rho in autotune.RHOS:
            work.launch(tri.MAP_LAMBDA, rho)
    assert [c[0] for c in calls] == ["tri_edm"] * 3 + ["tri_ca_step_tile"] * 3 + ["tet_at_energy"] * 3
    assert all(c[2]["reg"] == 4 and c[2]["rho"] == r for c, r in zip(calls[:3], autotune.RHOS))
    assert all(c[2]["rho"] == r for c, r in zip(calls[3:6], autotune.RHOS))
