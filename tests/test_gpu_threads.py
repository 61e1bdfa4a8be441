"""Handles of different sizes and options on several host threads, one handle each: every call is
accepted, whatever the other threads launch in between. The calls are made in a C loop, which the
interpreter's lock does not serialise."""
import ctypes
import shutil
import subprocess
import threading

import numpy as np
import pytest

from tests.gpu_common import rt_module, to_dev, torch_cuda

pytestmark = pytest.mark.gpu

LOOP = """
#include <stdint.h>
int scalings(int (*f)(void*, const double*), void* h, int n) {
    int bad = 0;
    for (int i = 0; i < n; ++i) bad += f(h, 0) != 0;
    return bad;
}
int steps(int (*f)(void*, uint64_t, int64_t), void* h, int64_t l, int n) {
    int bad = 0;
    for (int i = 0; i < n; ++i) bad += f(h, (uint64_t)i, l) != 0;
    return bad;
}
"""


@pytest.fixture(scope="module")
def loop(tmp_path_factory):
    cc = shutil.which("gcc") or shutil.which("cc")
    if cc is None:
        pytest.skip("no host C compiler")
    d = tmp_path_factory.mktemp("loop")
    (d / "loop.c").write_text(LOOP)
    subprocess.run([cc, "-O2", "-shared", "-fPIC", str(d / "loop.c"), "-o", str(d / "loop.so")], check=True)
    return ctypes.CDLL(str(d / "loop.so"))


def _on_threads(torch, handles, call):
    """call(handle) on a thread each; the refused calls of every thread."""
    bad = [None] * len(handles)

    def work(i):
        bad[i] = call(handles[i])

    threads = [threading.Thread(target=work, args=(i,)) for i in range(len(handles))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    return bad


def test_slicing_with_other_digit_counts(loop):
    torch, rt = torch_cuda(), rt_module()
    fn = ctypes.cast(rt.load_library().rtproj_set_scaling, ctypes.c_void_p)
    A = to_dev(torch, np.random.default_rng(1).standard_normal((64, 2048)))
    counts = [6, 7, 6, 7, 8, 10]
    names = ("sketch_slices", "gram_slices", "gram2_slices", "apply_slices", "resid_slices")
    P = [rt.Projector(A, l_max=70, k_max=1, stream=torch.cuda.Stream(), async_=1, scalable=1, **{n: s for n in names})
         for s in counts]
    assert _on_threads(torch, P, lambda p: loop.scalings(fn, p._h, 2000)) == [0] * len(P)
    assert [p.info()["status"] for p in P] == [0] * len(P)


def test_dense_steps_of_other_sizes(loop):
    torch, rt = torch_cuda(), rt_module()
    fn = ctypes.cast(rt.load_library().rtproj_precondition, ctypes.c_void_p)
    rng = np.random.default_rng(2)
    P = [rt.Projector(to_dev(torch, rng.standard_normal((m, 16 * m))), l_max=2 * m + 8, k_max=1, mode=mode,
                      stream=torch.cuda.Stream(), async_=1)
         for m, mode in ((40, "mixed"), (128, "mixed"), (180, "mixed"), (150, "fp64"))]
    assert _on_threads(torch, P, lambda p: loop.steps(fn, p._h, ctypes.c_int64(p.l_max), 60)) == [0] * len(P)
    assert [p.info()["status"] for p in P] == [0] * len(P)


def test_sparse_steps_of_other_ranks(loop):
    torch, rt = torch_cuda(), rt_module()
    fn = ctypes.cast(rt.load_library().rtproj_precondition, ctypes.c_void_p)
    rng = np.random.default_rng(3)
    m, n = 48, 2000
    rp = np.arange(m + 1, dtype=np.int64) * 125
    ci = np.concatenate([np.sort(rng.choice(n, 125, replace=False)) for _ in range(m)]).astype(np.int32)
    v = rng.standard_normal(ci.size)
    P = [rt.SparseProjector(to_dev(torch, rp), to_dev(torch, ci), to_dev(torch, v), n, U=to_dev(torch, rng.standard_normal((m, r))),
                            V=to_dev(torch, rng.standard_normal((r, n)) / 64), l_max=m + 4, k_max=1,
                            stream=torch.cuda.Stream(), async_=1) for r in (1, 8, 24, 48)]
    assert _on_threads(torch, P, lambda p: loop.steps(fn, p._h, ctypes.c_int64(p.l_max), 150)) == [0] * len(P)
    assert [p.info()["status"] for p in P] == [0] * len(P)
