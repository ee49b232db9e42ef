"""Which weights choose: those that rank the present classes; the first ones,
trained when the default was the tiles, choose nothing.  (No GPU: parameters for
other classes are not evaluated.)"""
import json

import numpy as np
import pytest

torch = pytest.importorskip("torch")


def _selector():
    from paper_1504_06474_gb300 import selector
    return selector


def test_weights_for_other_classes_choose_the_default():
    S = _selector()
    first = S.load_default()
    assert first is not None and not S.ranks_classes(first)
    X = np.random.default_rng(0).random((7, S.F)).astype(np.float32)
    assert np.array_equal(S.select(first, X, None), np.zeros(7))
    o = S.choose_opts(None, 1000, 1000, 5000, first)
    d = S.class_opts(0)
    assert [getattr(o, f) for f, _ in o._fields_] == [getattr(d, f) for f, _ in d._fields_]
    # copies still know what they rank, an array of a user's own does not say
    assert not S.ranks_classes(first.copy())
    assert S.ranks_classes(np.asarray(first, np.float32).view(np.ndarray))


def test_current_weights_rank_the_classes():
    S = _selector()
    now = S.load_current()
    assert now is not None and S.ranks_classes(now)
    assert list(now.classes) == [c[0] for c in S.CLASSES]
    assert now.size == S.F * S.H1 + S.H1 + S.H1 * S.H2 + S.H2 + S.H2 * S.K + S.K
    assert np.all(np.isfinite(now))
    t = torch.as_tensor(now)
    assert t.dtype == torch.float32 and t.numel() == now.size


def test_a_file_for_other_classes_is_not_current(tmp_path, monkeypatch):
    S = _selector()
    with open(S.CURRENT_WEIGHTS) as f:
        d = json.load(f)
    d["classes"][0] = "something else"
    p = tmp_path / "w.json"
    p.write_text(json.dumps(d))
    monkeypatch.setattr(S, "CURRENT_WEIGHTS", str(p))
    assert S.load_current() is None
    d["classes"] = [c[0] for c in S.CLASSES]
    p.write_text(json.dumps(d))
    assert S.load_current() is not None


@pytest.mark.gpu
@pytest.mark.parametrize("name", ["stencil160", "rmat20"])
def test_the_choice_is_no_slower_than_the_default(name):
    import synth
    from paper_1504_06474_gb300 import _build
    from paper_1504_06474_gb300 import ssspmv as C
    S = _selector()
    _build.build()
    dev = torch.device("cuda:0")
    A, x = synth.workload(name)
    Ad = S.to_device(A, x, dev)
    timer = S.Timer(dev)
    ms = []
    for opts in (S.choose_opts(Ad.rp, A.m, A.n, A.nnz, S.load_current()), S.class_opts(0)):
        ws = timer.workspace(max(256, C.ssspmv_workspace_bytes(A.m, A.nnz, 8, opts)))
        ms.append(timer.time_ms(lambda: C.check(C.ssspmv_csr_f64(
            A.m, A.n, A.nnz, Ad.rp, Ad.col, Ad.val, Ad.x, Ad.y, opts=opts, workspace=ws), "csr"), 9))
    assert ms[0] <= 1.05 * ms[1], ms
