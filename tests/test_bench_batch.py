"""bench.py's batched alpha sweep on CPU with stand-ins for the GPU: it runs on
per-phase launches, and an error of it ends the run."""
import ast
import inspect
import types

import pytest

import bench
from paper_2306_01959_gb300 import workloads as wl


class _Event:
    def __init__(self, **kw):
        pass

    def record(self, stream):
        pass

    def elapsed_time(self, other):
        return 1000.0


def _run(fail=False):
    made = []

    class Sim:
        stream, n = None, 100

        def __init__(self, cases, **kw):
            self.cases = cases
            made.append(kw)

        def step(self, dt, n):
            pass

        def sync(self):
            if fail:
                raise RuntimeError("device error")

        def close(self):
            pass

    torch = types.SimpleNamespace(cuda=types.SimpleNamespace(Event=_Event, synchronize=lambda: None))
    return made, lambda: bench.run_batch(None, types.SimpleNamespace(Simulation=Sim, MIXED=1), wl, torch, 0, 1)


def test_batch_runs_on_per_phase_launches():
    made, run = _run()
    out = run()
    assert len(made) == 65 and not any(kw.get("persistent") for kw in made)
    assert out["value"] == 100 * 1000.0 and out["speedup"] == 1.0


def test_an_error_of_the_batch_ends_the_run():
    _, run = _run(fail=True)
    with pytest.raises(RuntimeError):
        run()
    tree = ast.parse(inspect.getsource(bench.run_ours))
    guarded = [n for t in ast.walk(tree) if isinstance(t, ast.Try) for n in ast.walk(t)]
    assert not [n for n in guarded if isinstance(n, ast.Name) and n.id == "run_batch"]
