"""What the library's host code makes of device memory that runs out, without a
GPU: it runs against a stand-in CUDA runtime (fake_cudart.c), in which kernels
do nothing and any allocation can be made to fail. A failed call frees the
buffers it was growing, so nothing that stood on them may be used afterwards:
no tree, no node capacity, no captured step."""
import ctypes
import json
import os
import subprocess
import sys

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)

PRELUDE = """
import ctypes, json, sys
sys.path.insert(0, {root!r})
from paper_1502_07442_gb300 import binding as ng
F = ctypes.CDLL({fake!r})
F.fake_set_limit.argtypes = [ctypes.c_size_t]
F.fake_fail_at.argtypes = [ctypes.c_long]
for f in ("fake_in_use", "fake_live", "fake_mallocs", "fake_captures", "fake_replays"):
    getattr(F, f).restype = ctypes.c_size_t
L = ng.lib()
vp, i64 = ctypes.c_void_p, ctypes.c_int64
def params(leaf=8):
    p = ng.NgParams()
    p.D, p.box, p.eps, p.asmth, p.rcut_over_rs = 1, 1.0, 1e-4, 0.02, 4.5
    p.theta, p.leaf_size, p.G[0][0] = 0.5, leaf, 1.0
    return p
def context(**k):
    c = vp()
    p = params(**k)
    assert L.ng_create(ctypes.byref(c), ctypes.byref(p), None) == ng.NG_OK
    return c
def state(n):
    # "device" arrays: pos, vel, type, mass, acc
    return [ctypes.cast(ctypes.create_string_buffer(max(1, b * n)), vp) for b in (24, 12, 1, 4, 12)]
def build(c, n, s):
    return L.ng_build_tree(c, i64(n), s[0], s[2], s[3], None, None)
def step(c, n, s, valid, k):
    return L.ng_step(c, i64(n), s[0], s[1], s[2], s[3], s[4], valid, k, ctypes.c_double(0.25))
"""


@pytest.fixture(scope="module")
def run(tmp_path_factory):
    from paper_1502_07442_gb300 import build
    build.build()
    d = tmp_path_factory.mktemp("fake")
    fake = str(d / "fake_cudart.so")
    subprocess.check_call(["gcc", "-O1", "-shared", "-fPIC", os.path.join(HERE, "fake_cudart.c"), "-o", fake])

    def go(body):
        script = d / "case.py"
        script.write_text(PRELUDE.format(root=ROOT, fake=fake) + body)
        r = subprocess.run([sys.executable, str(script)], capture_output=True, text=True, timeout=120,
                           env=dict(os.environ, LD_PRELOAD=fake))
        assert r.returncode == 0, r.stderr[-2000:]
        return json.loads(r.stdout.splitlines()[-1])
    return go


def test_a_failed_step_leaves_no_tree_and_no_capacity(run):
    """Every allocation of a larger step fails in turn: the tree of the build
    before is then refused, and the next build holds all of its buffers again."""
    out = run("""
s, big = state(1000), state(50000)
rows = []
for k in range(200):
    c = context()
    assert build(c, 1000, s) == ng.NG_OK and L.ng_tree_force(c, s[4], None) == ng.NG_OK
    live = F.fake_live()
    F.fake_fail_at(k)
    r = step(c, 50000, big, 1, 1)
    F.fake_fail_at(-1)
    if r == ng.NG_OK:
        break
    refused = L.ng_tree_force(c, s[4], None)
    again = build(c, 1000, s), L.ng_tree_force(c, s[4], None)
    rows.append([r, refused, again[0], again[1], F.fake_live() >= live])
    L.ng_destroy(c)
print(json.dumps(dict(rows=rows, enomem=ng.NG_ENOMEM, estate=ng.NG_ESTATE)))
""")
    assert len(out["rows"]) > 30
    for k, r in enumerate(out["rows"]):
        assert r == [out["enomem"], out["estate"], 0, 0, True], (k, r)


@pytest.mark.parametrize("k", [0, 1, 5, 12])
def test_a_failed_batch_step_drops_the_captured_one(run, k):
    """A larger batch step whose k-th allocation fails has freed buffers that the
    step captured before reads: the next step at the old sizes is captured anew."""
    out = run(f"""
S, n = 2, 1000
b = vp()
P = (ng.NgParams * S)(params(), params())
assert L.ng_batch_create(ctypes.byref(b), S, P, None) == ng.NG_OK
st, big = [state(n), state(n)], [state(60000), state(n)]
def go(ns, states, valid, steps):
    arr = [(vp * S)(*[x[j].value for x in states]) for j in range(5)]
    return L.ng_batch_step(b, (i64 * S)(*ns), arr[0], arr[1], arr[2], arr[3], arr[4], valid, steps,
                           ctypes.c_double(0.25))
assert go([n, n], st, 0, 3) == ng.NG_OK
c1 = F.fake_captures()
assert go([n, n], st, 1, 3) == ng.NG_OK
c2 = F.fake_captures()
F.fake_fail_at({k})
r = go([60000, n], big, 0, 3)
F.fake_fail_at(-1)
assert go([n, n], st, 1, 3) == ng.NG_OK
print(json.dumps(dict(reused=c2 == c1, failed=r == ng.NG_ENOMEM, anew=F.fake_captures() > c2)))
""")
    assert out == dict(reused=True, failed=True, anew=True)


def test_a_slot_without_tables_is_configured_again(run):
    """A served request whose law tables could not be had fails; the next one with
    the same parameters does not run on what is left of them."""
    out = run("""
s = vp()
assert L.ng_serve_create(ctypes.byref(s), 1, ctypes.c_size_t(1 << 32)) == ng.NG_OK
n = 1000
a = state(n)
q = ng.NgRequest()
q.kind, q.n, q.params = 0, n, params()
q.params.D = 5                      # a larger table than the slot's first one
q.pos, q.type, q.mass, q.acc_out = [x.value for x in (a[0], a[2], a[3], a[4])]
res = (ng.NgResult * 1)()
def serve():
    assert L.ng_serve(s, ctypes.byref(q), res, 1, None, ctypes.c_double(30.0)) == ng.NG_OK
    return res[0].status
F.fake_fail_at(0)
first = serve()
F.fake_fail_at(-1)
second = serve()
reconf = i64()
L.ng_serve_stats(s, None, None, None, ctypes.byref(reconf))
print(json.dumps(dict(first=first == ng.NG_ENOMEM, second=second, configured=reconf.value)))
""")
    assert out == dict(first=True, second=0, configured=1)


def test_records_are_given_back_before_a_call_runs_out(run):
    """A step on 131072 bodies keeps its optional records (64 bytes a body); a later
    build that fits only without them gets their memory, and so does a batch
    member from another's."""
    out = run("""
n1, n2 = 131072, 4000000
s1, s2 = state(n1), state(n2)
def single(limit):
    F.fake_set_limit(limit)
    c = context()
    assert step(c, n1, s1, 1, 2) == ng.NG_OK
    held = F.fake_in_use()
    r = build(c, n2, s2), L.ng_tree_force(c, s2[4], None)
    top = F.fake_in_use()
    L.ng_destroy(c)
    return held, r, top
def batch(limit):
    F.fake_set_limit(limit)
    b = vp()
    P = (ng.NgParams * 2)(params(), params())
    assert L.ng_batch_create(ctypes.byref(b), 2, P, None) == ng.NG_OK
    def go(ns, states):
        arr = [(vp * 2)(*[x[j].value for x in states]) for j in range(5)]
        return L.ng_batch_step(b, (i64 * 2)(*ns), arr[0], arr[1], arr[2], arr[3], arr[4], 0, 2, ctypes.c_double(0.25))
    small = state(1000)
    assert go([n1, 1000], [s1, small]) == ng.NG_OK
    held = F.fake_in_use()
    r = [go([n1, n2], [s1, s2])]
    top = F.fake_in_use()
    L.ng_batch_destroy(b)
    return held, r, top
rows = []
for f, records in ((single, 64 * n1), (batch, 32 * n1)):
    held, r, top = f(1 << 30)
    tight = f(top - records // 2)
    rows.append([list(r), list(tight[1]), tight[0] == held, top - tight[2] == records])
print(json.dumps(rows))
""")
    assert out == [[[0, 0], [0, 0], True, True], [[0], [0], True, True]]


@pytest.mark.parametrize("call,size", [("build(c, n, s)", 32), ("step(c, n, s, 1, 1)", 64)])
def test_records_are_a_small_part_of_the_free_memory(run, call, size):
    """Taken only where 2048 bytes a body are free: 3 % of it at most."""
    out = run(f"""
n = 150000
s = state(n)
use = []
for limit in (1 << 33, 1 << 28):
    F.fake_set_limit(limit)
    c = context()
    assert {call} == ng.NG_OK
    use.append(F.fake_in_use())
    L.ng_destroy(c)
print(json.dumps(use[0] - use[1]))
""")
    assert out == size * 150000
