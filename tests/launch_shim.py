"""A stand-in for cudaLaunchKernelExC, preloaded into a child process: it can
refuse the n-th launch from now (an error code, nothing is launched) and
lists the names of the kernels that were launched."""

import os
import subprocess
import sys
import textwrap

SOURCE = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stdio.h>
#include <string.h>

typedef int (*launch_fn)(const void *, const void *, void **);
typedef int (*name_fn)(const char **, const void *);
static long refuse_at, count;
static char names[1 << 20];

void shim_refuse(long n) { refuse_at = n; count = 0; }
void shim_forget(void) { names[0] = 0; }
const char *shim_names(void) { return names; }

int cudaLaunchKernelExC(const void *config, const void *func, void **args)
{
    void *rt = dlopen("libcudart.so.13", RTLD_LAZY | RTLD_NOLOAD);
    const char *name = "";
    ((name_fn)dlsym(rt, "cudaFuncGetName"))(&name, func);
    if (strlen(names) + strlen(name) + 2 < sizeof names) strcat(strcat(names, name), "\n");
    if (++count == refuse_at) return 701;  /* cudaErrorLaunchOutOfResources */
    return ((launch_fn)dlsym(rt, "cudaLaunchKernelExC"))(config, func, args);
}
"""


def run_child(tmp_path, body: str) -> str:
    """Run `body` (which finds `shim`, `dm`, `np`, `inputs`) in a child with
    the stand-in; returns its output."""
    src, lib = tmp_path / "shim.c", tmp_path / "libshim.so"
    src.write_text(SOURCE)
    subprocess.run(["gcc", "-O1", "-shared", "-fPIC", "-o", str(lib), str(src), "-ldl"], check=True)
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    head = f"""
        import ctypes
        import numpy as np
        from paper_1511_04633_gb300 import dmrt as dm, inputs
        shim = ctypes.CDLL({str(lib)!r})
        shim.shim_refuse.argtypes = [ctypes.c_long]
        shim.shim_names.restype = ctypes.c_char_p
    """
    code = textwrap.dedent(head) + textwrap.dedent(body)
    env = dict(os.environ, LD_PRELOAD=str(lib), PYTHONPATH=root)
    r = subprocess.run([sys.executable, "-c", code], cwd=root, env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-3000:]
    return r.stdout
