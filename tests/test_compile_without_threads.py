"""Compilation where the system gives no threads: an FP64 model's two modules one after the other, and no
exception through the C entry."""
import os
import subprocess
import sys

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHIM = r'''
#define _GNU_SOURCE
#include <dlfcn.h>
#include <errno.h>
#include <pthread.h>
#include <stdlib.h>
int pthread_create(pthread_t *t, const pthread_attr_t *a, void *(*f)(void *), void *p) {
    if (getenv("NO_MORE_THREADS")) return EAGAIN;
    int (*next)(pthread_t *, const pthread_attr_t *, void *(*)(void *), void *) = dlsym(RTLD_NEXT, "pthread_create");
    return next(t, a, f, p);
}
'''
RUN = r'''
import os
from paper_2608_16265_gb300 import binding
from paper_2608_16265_gb300.ir import Model, sin
m = Model()
x = m.add_var(5)
m.add_con(lambda d: sin(x[d.k]) * x[d.k + 1], n=4)
flat = m.flat()
binding.load()
os.environ["NO_MORE_THREADS"] = "1"
binding.exa_compile_check(flat, block=64)
print("compiled")
'''


def test_compile_without_threads(tmp_path):
    (tmp_path / "shim.c").write_text(SHIM)
    so = str(tmp_path / "shim.so")
    subprocess.run(["gcc", "-shared", "-fPIC", "-o", so, str(tmp_path / "shim.c"), "-ldl"], check=True)
    r = subprocess.run([sys.executable, "-c", RUN], cwd=ROOT, capture_output=True, text=True,
                       env=dict(os.environ, LD_PRELOAD=so, PYTHONPATH=ROOT))
    assert r.returncode == 0 and "compiled" in r.stdout, r.stderr[-2000:]
