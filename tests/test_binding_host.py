"""Host side of the Python binding: what needs no GPU."""
import os
import subprocess
import sys
import threading

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def b2():
    from paper_2411_07211_b200 import build
    build.build()
    from paper_2411_07211_b200 import binding
    return binding


def test_recordings_of_two_threads_stay_apart(b2):
    """Two prepare() calls whose thunks overlap, the first to begin also the first to end: what a thread hands to its
    recording ends up in that one, and with both over nothing is recorded any more."""
    began, both, first_over = threading.Event(), threading.Event(), threading.Event()
    mine = {"a": object(), "b": object(), "after": object()}
    held = lambda: [sys.getrefcount(mine[k]) for k in ("a", "b", "after")]
    base = held()
    over = lambda: [n - m for n, m in zip(held(), base)]  # references taken since then
    replays = {}

    def a():
        began.set()
        assert both.wait(20)
        b2._native.keep(mine["a"])

    def b():
        assert began.wait(20)
        both.set()
        assert first_over.wait(20)
        b2._native.keep(mine["b"])

    def run(name, thunk, done=None):
        replays[name] = b2.prepare(thunk)
        if done:
            done.set()

    threads = [threading.Thread(target=run, args=("a", a, first_over)), threading.Thread(target=run, args=("b", b))]
    for t in threads:
        t.start()
    for t in threads:
        t.join(30)
    assert set(replays) == {"a", "b"}
    b2._native.keep(mine["after"])  # (no recording runs: nothing may hold on to it)
    assert over() == [1, 1, 0]
    del replays["a"]
    assert over() == [0, 1, 0]
    del replays["b"]
    assert over() == [0, 0, 0]


def test_recordings_nest(b2):
    """A prepare() inside the thunk of another one, ended by an exception too, leaves the outer recording in place."""
    inner, outer = object(), object()
    base = sys.getrefcount(inner), sys.getrefcount(outer)
    got = []

    def fails():
        raise RuntimeError("stop")

    def thunk():
        got.append(b2.prepare(lambda: b2._native.keep(inner)))
        with pytest.raises(RuntimeError, match="stop"):
            b2.prepare(fails)
        b2._native.keep(outer)

    replay = b2.prepare(thunk)
    assert (sys.getrefcount(inner) - base[0], sys.getrefcount(outer) - base[1]) == (1, 1)
    got.clear()
    assert (sys.getrefcount(inner) - base[0], sys.getrefcount(outer) - base[1]) == (0, 1)
    del replay
    assert sys.getrefcount(outer) == base[1]


def test_the_reason_why_the_module_does_not_load_is_told(b2):
    """Importing the package works without the compiled module; the first call says what the import said."""
    code = """
import sys
class Refuse:
    def find_spec(self, name, path=None, target=None):
        if name.endswith('._binding'):
            raise ImportError('undefined symbol: _ZN3c10')
sys.meta_path.insert(0, Refuse())
from paper_2411_07211_b200 import binding as b2
for call in (lambda: b2.axpy(None, 1, 1.0, None, 1, None, 1), lambda: b2.prepare(lambda: None)):
    try:
        call()
    except ImportError as e:
        assert 'undefined symbol: _ZN3c10' in str(e) and isinstance(e.__cause__, ImportError), e
    else:
        raise AssertionError('no error')
print('told')
"""
    res = subprocess.run([sys.executable, "-c", code], cwd=ROOT, capture_output=True, text=True, timeout=300)
    assert res.returncode == 0 and "told" in res.stdout, res.stdout + res.stderr


def test_another_interpreter_or_torch_rebuilds_the_module(monkeypatch):
    from paper_2411_07211_b200 import build
    now, library = build._binding_digest(), build._digest()
    with monkeypatch.context() as m:
        m.setattr(build.importlib.metadata, "version", lambda name: "0.0")
        assert build._binding_digest() != now
    with monkeypatch.context() as m:
        m.setattr(sys, "version", "4.0")
        assert build._binding_digest() != now and build._digest() == library
    assert build._binding_digest() == now


def test_routines_describe_themselves(b2):
    """Name, docstring, signature and pickling, as Python functions have them."""
    import copy
    import inspect
    import pickle
    for name in b2._NAMES:
        f = getattr(b2, name)
        sig = inspect.signature(f)
        assert list(sig.parameters)[0] == "ctx" and sig.parameters["check"].default is True
        assert f.__name__ == name and inspect.getdoc(f)
        assert pickle.loads(pickle.dumps(f)) is f and copy.deepcopy(f) is f
        if name != "rotm":  # (a Python function around the native one)
            assert f.__doc__.startswith(f"{name}{sig}") and f.__qualname__ == name
    assert list(inspect.signature(b2.gemv).parameters) == ["ctx", "order", "trans", "m", "n", "alpha", "a", "lda", "x", "incx",
                                                           "beta", "y", "incy", "check"]
    inspect.signature(b2.trsv).bind(1, 2, 3, 4, 5, 6, "a", 7, x="x", incx=1)
    with pytest.raises(TypeError):
        inspect.signature(b2.copy).bind(1, 2)
