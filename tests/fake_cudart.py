"""A stand-in for the CUDA runtime, for tests of the host code without a GPU: device memory is host memory, kernels do
nothing and are recorded.  ``run_child`` runs Python code in a child process whose library calls go to it."""
import os
import shutil
import subprocess
import sys

import pytest

from paper_1801_04382_gb300 import build as pkg_build

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include <stdio.h>
#include <stdlib.h>
#include <string.h>
typedef int E; typedef void *P; typedef size_t Z;
typedef struct { unsigned x, y, z; } D3;
typedef struct { int id; char pad[4]; union { char pad[64]; int cooperative; D3 cluster; } v; } Attr;
typedef struct { D3 grid, block; Z smem; P stream; Attr *attrs; unsigned n; } Config;
static int left = -1, made = 0, launches = 0, n_fun = 0;
static Z total = (Z)8 << 30, used = 0;
static struct { const void *host; const char *name; } fun[1024];
static char *log_ = 0;
static Z log_n = 0, log_cap = 0;
static Config pushed;
void fake_fail_in(int n) { left = n; }
int fake_mallocs(void) { return made; }
int fake_launches(void) { return launches; }
void fake_set_total(Z n) { total = n; }
const char *fake_log(void) { return log_ ? log_ : ""; }
void fake_log_clear(void) { log_n = 0; if (log_) *log_ = 0; }
static E launch(const void *f, const Config *c)
{
  const char *name = "?";
  int coop = 0, cluster = 1;
  for (int i = 0; i < n_fun; ++i) if (fun[i].host == f) name = fun[i].name;
  for (unsigned i = 0; i < c->n; ++i) {
    if (c->attrs[i].id == 2) coop = c->attrs[i].v.cooperative;
    if (c->attrs[i].id == 4) cluster = (int)c->attrs[i].v.cluster.x;
  }
  if (log_n + 1024 > log_cap) log_ = realloc(log_, log_cap = log_cap * 2 + 65536);
  log_n += (Z)snprintf(log_ + log_n, 1024, "%s %u %u %zu %d %d\n", name, c->grid.x, c->block.x, c->smem, coop, cluster);
  ++launches;
  return 0;
}
E cudaMalloc(P *p, Z n)
{
  *p = 0;
  if ((left > 0 && --left == 0) || used + n > total) return 2;
  Z *h = calloc(1, n + 256);
  if (!h) return 2;
  ++made;
  used += *h = n;
  *p = (char *)h + 256;
  return 0;
}
E cudaFree(P p) { if (p) { Z *h = (Z *)((char *)p - 256); used -= *h; free(h); } return 0; }
E cudaMemcpy(P d, const void *s, Z n, int k) { (void)k; if (n && (!d || !s)) return 1; memcpy(d, s, n); return 0; }
E cudaMemcpyAsync(P d, const void *s, Z n, int k, P st) { (void)st; return cudaMemcpy(d, s, n, k); }
E cudaMemsetAsync(P d, int v, Z n, P st) { (void)st; if (n && !d) return 1; memset(d, v, n); return 0; }
E cudaMemGetInfo(Z *f, Z *t) { *t = total; *f = total - used; return 0; }
E cudaGetDevice(int *d) { *d = 0; return 0; }
E cudaDeviceGetAttribute(int *v, int a, int d) { (void)a; (void)d; *v = 152; return 0; }
E cudaGetLastError(void) { return 0; }
const char *cudaGetErrorString(E e) { (void)e; return "stand-in"; }
E cudaFuncSetAttribute(const void *f, int a, int v) { (void)f; (void)a; (void)v; return 0; }
E cudaOccupancyMaxActiveBlocksPerMultiprocessorWithFlags(int *n, const void *f, int b, Z s, unsigned g)
{ (void)f; (void)b; (void)s; (void)g; *n = 2; return 0; }
E cudaGetSymbolAddress(P *p, const void *s) { (void)s; static char mem[1 << 20]; *p = mem; return 0; }
E cudaStreamSynchronize(P s) { (void)s; return 0; }
E cudaStreamCreateWithFlags(P *s, unsigned f) { (void)f; *s = malloc(1); return 0; }
E cudaStreamDestroy(P s) { free(s); return 0; }
E cudaStreamWaitEvent(P s, P e, unsigned f) { (void)s; (void)e; (void)f; return 0; }
E cudaStreamBeginCapture(P s, int m) { (void)s; (void)m; return 0; }
E cudaStreamEndCapture(P s, P *g) { (void)s; *g = malloc(1); return 0; }
E cudaGraphCreate(P *g, unsigned f) { (void)f; *g = malloc(1); return 0; }
E cudaGraphDestroy(P g) { free(g); return 0; }
E cudaGraphExecDestroy(P g) { free(g); return 0; }
E cudaGraphInstantiate(P *x, P g, unsigned long long f) { (void)g; (void)f; *x = malloc(1); return 0; }
E cudaGraphLaunch(P x, P s) { (void)x; (void)s; return 0; }
E cudaGraphAddChildGraphNode(P *n, P g, const P *d, Z k, P c) { (void)g; (void)d; (void)k; (void)c; *n = 0; return 0; }
E cudaGraphGetNodes(P g, P *n, Z *k) { (void)g; (void)n; *k = 0; return 0; }
E cudaEventCreate(P *s) { *s = malloc(1); return 0; }
E cudaEventCreateWithFlags(P *s, unsigned f) { (void)f; *s = malloc(1); return 0; }
E cudaEventDestroy(P s) { free(s); return 0; }
E cudaEventRecord(P e, P s) { (void)e; (void)s; return 0; }
E cudaEventSynchronize(P e) { (void)e; return 0; }
E cudaEventElapsedTime(float *ms, P a, P b) { (void)a; (void)b; *ms = 1; return 0; }
E cudaLaunchKernelExC(const Config *c, const void *f, P *a) { (void)a; return launch(f, c); }
E __cudaPushCallConfiguration(D3 g, D3 b, Z s, P st) { Config c = {g, b, s, st, 0, 0}; pushed = c; return 0; }
E __cudaPopCallConfiguration(D3 *g, D3 *b, Z *s, P st) { *g = pushed.grid; *b = pushed.block; *s = pushed.smem; *(P *)st = pushed.stream; return 0; }
E __cudaLaunchKernel(P k, D3 g, D3 b, P *a, Z s, P st) { (void)a; Config c = {g, b, s, st, 0, 0}; return launch(k, &c); }
E __cudaGetKernel(P *k, const void *f) { *k = (P)f; return 0; }
P *__cudaRegisterFatBinary(P f) { (void)f; static P h; return &h; }
void __cudaRegisterFatBinaryEnd(P *h) { (void)h; }
void __cudaRegisterFunction(P *h, const void *host, char *d, const char *name) { (void)h; (void)d; if (n_fun < 1024) { fun[n_fun].host = host; fun[n_fun++].name = name; } }
void __cudaRegisterVar(void) {}
void __cudaUnregisterFatBinary(P *h) { (void)h; }
"""


def run_child(tmp_path, code, *args):
    """Run ``code`` (sys.argv[1]: the stand-in's path, then ``args``); it has to print "ok" and nothing else."""
    if not shutil.which("gcc"):
        pytest.skip("no C compiler")
    if not os.path.exists(pkg_build.lib_path()):
        pkg_build.build()
    src, so = tmp_path / "fake_cudart.c", tmp_path / "libfake_cudart.so"
    src.write_text(SOURCE)
    subprocess.run(["gcc", "-shared", "-fPIC", "-O1", "-w", str(src), "-o", str(so)], check=True)
    env = dict(os.environ, LD_PRELOAD=str(so), PYTHONPATH=ROOT)
    res = subprocess.run([sys.executable, "-c", code, str(so), *[str(a) for a in args]], env=env, capture_output=True,
                         text=True, timeout=300)
    assert res.returncode == 0 and res.stdout.strip() == "ok", res.stdout + res.stderr
