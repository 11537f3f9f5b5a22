"""alp_set_wait_timeout_ms against the first use of the limit: a limit set
while the library reads its default from the environment is the one that
holds.  A C program (its own getenv sets the limit, as another thread may at
that moment) loads the library, so the order is fixed and no GPU is needed."""
import os
import subprocess

import pytest

PROGRAM = r"""
#define _GNU_SOURCE
#include <dlfcn.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>
extern char** environ;
static int (*set_limit)(double);
static double wanted;

char* getenv(const char* name) {
    if (set_limit && wanted > 0 && !strcmp(name, "ALP_WAIT_TIMEOUT_MS")) set_limit(wanted);
    const size_t n = strlen(name);
    for (char** e = environ; *e; ++e)
        if (!strncmp(*e, name, n) && (*e)[n] == '=') return *e + n + 1;
    return 0;
}

int main(int argc, char** argv) {
    void* lib = dlopen(argv[1], RTLD_NOW);
    if (!lib) return fprintf(stderr, "%s\n", dlerror()), 2;
    uint64_t (*limit)(void) = (uint64_t (*)(void))dlsym(lib, "_ZN3alp15wait_timeout_nsEv");
    set_limit = (int (*)(double))dlsym(lib, "alp_set_wait_timeout_ms");
    if (!limit || !set_limit) return 3;
    if (argc > 2) sscanf(argv[2], "%lf", &wanted);
    const unsigned long long first = limit(), second = limit();
    printf("%llu %llu\n", first, second);
    return 0;
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("limit")
    src, exe = d / "limit.c", d / "limit"
    src.write_text(PROGRAM)
    subprocess.run(["gcc", "-O1", "-rdynamic", "-o", str(exe), str(src), "-ldl"], check=True)
    return str(exe)


@pytest.mark.parametrize("env,wanted,ns", [
    (None, None, 4000_000_000), ("70", None, 70_000_000),     # the default, the environment's
    (None, "250", 250_000_000), ("70", "250", 250_000_000)])  # set meanwhile
def test_limit_set_while_the_default_is_read(alp, program, env, wanted, ns):
    e = {k: v for k, v in os.environ.items() if k != "ALP_WAIT_TIMEOUT_MS"}
    if env is not None:
        e["ALP_WAIT_TIMEOUT_MS"] = env
    r = subprocess.run([program, alp.LIB_PATH] + ([wanted] if wanted else []), env=e,
                       capture_output=True, text=True, timeout=120)
    assert r.returncode == 0, r.stderr
    assert r.stdout.split() == [str(ns), str(ns)]
