"""The order of streams in the serving loop, without a GPU: runs are created
on the admission stream, where sdm_set_attributes leaves the kernels that
write their layout and record running, so the stream that steps them has to
wait for that stream first, at every batch that takes new runs."""
import numpy as np
import torch

from paper_2103_17238_gb300 import inputs as I
from paper_2103_17238_gb300 import serve


class _Stream:
    def __init__(self, log, name):
        self.log, self.name = log, name

    def wait_stream(self, other):
        self.log.append(("wait", self.name, other.name))


class _Event:
    def __init__(self, enable_timing=False):
        pass

    def record(self, stream):
        pass

    def synchronize(self):
        pass

    def elapsed_time(self, other):
        return 1.0


def test_steps_wait_for_the_admitted_runs(monkeypatch):
    log = []
    main, now = _Stream(log, "main"), []

    class _On:
        def __init__(self, stream):
            self.stream = stream

        def __enter__(self):
            now.append(self.stream)

        def __exit__(self, *exc):
            now.pop()

    class _Run:
        def spectrum(self, edges):
            return np.zeros(len(edges) - 1)

        def close(self):
            pass

    def make_run(inst):
        log.append(("create", now[-1].name if now else "main", inst.seed))
        return _Run()

    class _Batch:
        def __init__(self, runs, **kw):
            log.append(("batch", now[-1].name if now else "main", len(runs)))

        def step(self, k):
            log.append(("step", now[-1].name if now else "main", k))

        def close(self):
            pass

    monkeypatch.setattr(torch.cuda, "current_stream", lambda *a: main)
    monkeypatch.setattr(torch.cuda, "Stream", lambda *a, **k: _Stream(log, "admission"))
    monkeypatch.setattr(torch.cuda, "stream", _On)
    monkeypatch.setattr(torch.cuda, "Event", _Event)
    monkeypatch.setattr(serve, "make_run", make_run)
    monkeypatch.setattr(serve, "footprint", lambda inst: 1)
    monkeypatch.setattr(serve.sdm, "Batch", _Batch)

    def request(seed, steps):
        inst = I.box_golovin(64, seed=seed)
        inst.steps = steps
        return I.Request(1e-9 * seed, inst)

    out = serve.Server(10, chunk=4, admit_per_pass=2).serve([request(i, 4 * (i + 1)) for i in range(5)])
    assert out["requests"] == 5
    created, ready = 0, 0
    for what, where, arg in log:
        if what == "create":
            assert where == "admission"
            created += 1
        elif what == "wait":
            assert (where, arg) == ("main", "admission")
            ready = created
        elif what == "batch":
            assert where == "main" and ready == created, log  # (a batch's own work may touch the records)
        else:
            assert where == "main"
    assert created == 5 and any(w == "step" for w, _, _ in log)
