"""Pages of large host outputs: populating them changes no byte, starts no thread where the pages are there, and
leaves memory alone that it cannot populate.  Compiled from the library's own header."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

PROG = r'''
#include <stdio.h>
#include <string.h>
#include "host_pages.h"
static const size_t MB = 1 << 20, page = (size_t)sysconf(_SC_PAGESIZE);
static unsigned char* fresh(size_t n, int prot) {
  void* p = mmap(nullptr, n, prot, MAP_PRIVATE | MAP_ANONYMOUS, -1, 0);
  return p == MAP_FAILED ? nullptr : (unsigned char*)p;
}
static double present(unsigned char* p, size_t n) {
  std::vector<unsigned char> v(n / page);
  if (mincore(p, n, v.data()) != 0) return -1.0;
  size_t s = 0;
  for (unsigned char c : v) s += c & 1;
  return (double)s / v.size();
}
int main() {
  const size_t n = 48 * MB;
  // fresh memory at an odd address: the whole range becomes present and stays zero
  unsigned char* a = fresh(n, PROT_READ | PROT_WRITE);
  printf("%d", pb::populate_pages(a + 5, n - 11) > 0);
  printf(" %.3f", present(a, n));
  size_t bad = 0;
  for (size_t i = 0; i < n; ++i) bad += a[i] != 0;
  // used memory: nothing to do, nothing changed
  for (size_t i = 0; i < n; ++i) a[i] = (unsigned char)(i * 7 + 1);
  printf(" %d", pb::populate_pages(a + 5, n - 11));
  for (size_t i = 0; i < n; ++i) bad += a[i] != (unsigned char)(i * 7 + 1);
  // a half-used buffer keeps its contents
  unsigned char* b = fresh(n, PROT_READ | PROT_WRITE);
  memset(b, 9, n / 2);
  printf(" %d", pb::populate_pages(b, n) > 0);
  for (size_t i = 0; i < n; ++i) bad += b[i] != (i < n / 2 ? 9 : 0);
  // below the size, read-only, not mapped: left alone
  unsigned char* c = fresh(n, PROT_READ | PROT_WRITE);
  printf(" %d", pb::populate_pages(c, 31 * MB));
  printf(" %.3f", present(c, n));
  unsigned char* d = fresh(n, PROT_READ);
  pb::populate_pages(d, n);
  unsigned char* e = fresh(n, PROT_READ | PROT_WRITE);
  munmap(e, n);
  printf(" %d %zu\n", pb::populate_pages(e, n), bad);
  return 0; }'''


def test_populate_keeps_contents(tmp_path):
    src, exe = tmp_path / "p.cpp", tmp_path / "p"
    src.write_text(PROG)
    subprocess.check_call(["g++", "-O1", "-std=c++17", "-pthread", "-I",
                           os.path.join(ROOT, "paper_2510_23419_gb300", "csrc"), str(src), "-o", str(exe)])
    out = subprocess.check_output([str(exe)]).decode().split()
    assert out == ["1", "1.000", "0", "1", "0", "0.000", "0", "0"], out
