"""The host-thread loop of the set-up and of the potential's tree (parallel_for): every index runs once, an exception of
a body reaches the caller as itself instead of ending the process, and shares whose thread the system refuses to
start still run.  A small program around the header, with a pthread_create that can be told to fail."""
import os
import subprocess

import pytest

from paper_2306_11324_gb300 import build

SOURCE = r"""
#include <dlfcn.h>
#include <pthread.h>

#include <atomic>
#include <cerrno>
#include <cstdio>
#include <cstring>
#include <new>
#include <string>
#include <vector>

#include "internal.h"

static int allowed = 1 << 30;  // threads that still start
extern "C" int pthread_create(pthread_t *t, const pthread_attr_t *a, void *(*f)(void *), void *x) {
  using Fn = int (*)(pthread_t *, const pthread_attr_t *, void *(*)(void *), void *);
  static Fn real = reinterpret_cast<Fn>(dlsym(RTLD_NEXT, "pthread_create"));
  return allowed-- > 0 ? real(t, a, f, x) : EAGAIN;
}

int main(int argc, char **argv) {
  const std::string what = argv[1];
  const long n = 1000;
  std::vector<std::atomic<int>> hits(n);
  if (what == "threads") allowed = std::atoi(argv[2]);
  std::string got = "none";
  try {
    igabem::parallel_for(n, [&](long i) {
      hits[i]++;
      if (what == "memory" && i % 7 == 3) throw std::bad_alloc();
      if (what == "message" && i == 997) throw std::string("body");
    });
    igabem::parallel_for(0, [&](long) { hits[0] += 100; });
  } catch (const std::bad_alloc &) {
    got = "bad_alloc";
  } catch (const std::string &s) {
    got = s;
  }
  long once = 0;
  for (auto &h : hits) once += h == 1;
  std::printf("%s %ld\n", got.c_str(), once);
}
"""


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("threads")
    (d / "check.cpp").write_text(SOURCE)
    exe = d / "check"
    subprocess.run([build._nvcc(), "-std=c++17", "-I" + build.CSRC, "-I" + build.INCLUDE, str(d / "check.cpp"), "-o", str(exe),
                    "-Xcompiler", "-pthread", "-ldl", "-lpthread"], check=True)
    return str(exe)


def run(program, *args):
    r = subprocess.run([program, *args], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stderr
    return r.stdout.split()


def test_every_index_once(program):
    assert run(program, "plain") == ["none", "1000"]


def test_exception_of_a_body_reaches_the_caller(program):
    assert run(program, "memory")[0] == "bad_alloc"
    assert run(program, "message")[0] == "body"


@pytest.mark.parametrize("threads", [0, 1, 5])
def test_shares_without_a_thread_run_on_the_caller(program, threads):
    assert run(program, "threads", str(threads)) == ["none", "1000"]
