"""What the tuners time: the call without a tune among the candidates, and no
kernel twice (host logic, with the launches replaced by recorders)."""
import types

import pytest
import torch

import paper_2404_19638_gb300.autotune as at
from paper_2404_19638_gb300 import Batch, Item, OP_SDDMM, OP_SPMM


def _pattern(M, N, nnz):
    S = types.SimpleNamespace(M=M, N=N, nnz=nnz, device=torch.device("cpu"), has_schedule=True, vals=None,
                              rowptr=(torch.arange(M + 1) * nnz // M).int(), W=512)
    S.schedule_info = lambda: {"chunk_work": S.W}
    S.build_schedule = lambda W: setattr(S, "W", W)
    S.transpose_plan = lambda W=None: setattr(S, "W", W or S.W)
    return S


def _kernel(op, K, dtype, t):
    """The fields of a tune that its kernel reads."""
    t = {k: v for k, v in t.items() if k != "stages"}
    if t["variant"] == 2 and (op != "sddmm" or K % at._VEC[dtype]):
        t = {"variant": 2}
    return tuple(sorted(t.items()))


@pytest.mark.parametrize("op", ["sddmm", "spmm", "spmm_t"])
@pytest.mark.parametrize("dtype,K", [(torch.float32, 50), (torch.float32, 64), (torch.bfloat16, 128)])
def test_autotuner_times_each_kernel_once(monkeypatch, tmp_path, op, dtype, K):
    S = _pattern(40, 30, 200)
    calls = []
    monkeypatch.setattr(at, "ops", types.SimpleNamespace(**{n: lambda *a, tune, **k: calls.append(tune)
                                                            for n in ("sddmm", "spmm", "spmm_t")}))
    monkeypatch.setattr(at.Autotuner, "_time", lambda self, fn: (fn(), 1.0 - 1e-3 * len(calls))[1])
    tuner = at.Autotuner(cache_path=str(tmp_path / "c.json"), chunk_works=(256,))
    best = tuner.tune(S, op, torch.empty(40, K, dtype=dtype), torch.empty(30, K, dtype=dtype))
    assert {"variant": 2} in calls
    kernels = [_kernel(op, K, dtype, t) for t in calls]
    assert len(kernels) == len(set(kernels))
    assert best["tune"] == calls[-1]


def test_cache_entries_of_other_kernels_are_not_found(tmp_path):
    S = _pattern(40, 30, 200)
    tuner = at.Autotuner(cache_path=str(tmp_path / "c.json"))
    sig = at.pattern_signature(S.rowptr.numpy(), S.M, S.N)
    tuner._cache[f"{sig}|sddmm|float32|50"] = {"tune": {"variant": 2, "group_lanes": 16}, "chunk_work": 512, "ms": 1.0}
    assert tuner.lookup(S, "sddmm", torch.float32, 50) is None


def test_batch_tunes_shapes_of_sddmm_items_only(monkeypatch):
    """A batched SpMM item has one routine per row width: nothing to choose."""
    S = _pattern(40, 30, 200)
    A, B = torch.empty(40, 32), torch.empty(30, 32)
    b = Batch.__new__(Batch)
    b.items = [Item(OP_SDDMM, S, B, torch.empty(200), A=A), Item(OP_SPMM, S, B, torch.empty(40, 32))]
    b._tunes, b._h = [None, None], None
    tuned = []
    for name, f in (("_create", lambda self: None), ("_destroy", lambda self: None), ("__del__", lambda self: None),
                    ("_time", lambda self, reps: 1.0), ("set_registers", lambda self, r: None),
                    ("set_item_tune", lambda self, k, t: tuned.append((k, t)))):
        monkeypatch.setattr(Batch, name, f)
    b.autotune((64, 128), per_item=True)
    assert any(k == 0 and t is not None for k, t in tuned)
    assert all(t is None for k, t in tuned if k == 1)
