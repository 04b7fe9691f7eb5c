"""The serving loop when a finished request's result cannot be fetched: csrc/server.cu linked with
fakes of the solver calls it makes, so that a poll fails on the host without a device.  A batched
slot out of memory is polled again and keeps its result; any other failure ends the request as a
numerical error, never with a solved status beside vectors that were not filled."""
import os
import shutil
import subprocess

import pytest

from paper_2407_16144_gb300 import _build

pytestmark = pytest.mark.skipif(shutil.which("nvcc") is None and
                                not os.path.exists("/usr/local/cuda/bin/nvcc"),
                                reason="nvcc not available")

FAKES = r"""
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <chrono>
#include <thread>
#include "rhpdhg.h"

struct rhpdhg_batch { int status = -1, polls = 0; };
struct rhpdhg_handle { int polls = 0; };
static int first_rc, later_rc;            // codes of the first poll and of the ones after it

static int fake_poll(int polls, rhpdhg_result *r) {
  const int rc = polls == 1 ? first_rc : later_rc;
  r->status = RHPDHG_STATUS_OPTIMAL;      // filled before the failure, as a library may
  r->primal_obj = 7.0;
  if (rc == RHPDHG_OK) { r->x[0] = 3.0; r->y[0] = 4.0; }
  return rc;
}

extern "C" {
int64_t rhpdhg_batch_bytes_needed(const rhpdhg_problem *, int32_t) { return 1 << 20; }
int rhpdhg_batch_create(int32_t, int64_t, void *, rhpdhg_batch **b) {
  *b = new rhpdhg_batch;
  return RHPDHG_OK;
}
int rhpdhg_batch_add(rhpdhg_batch *b, const rhpdhg_problem *, const rhpdhg_params *, int32_t *s) {
  b->status = RHPDHG_STATUS_RUNNING;
  *s = 0;
  return RHPDHG_OK;
}
int rhpdhg_batch_step(rhpdhg_batch *b, int32_t) {
  b->status = RHPDHG_STATUS_OPTIMAL;
  return RHPDHG_OK;
}
int rhpdhg_batch_slot_status(const rhpdhg_batch *b, int32_t) { return b->status; }
int rhpdhg_batch_poll(rhpdhg_batch *b, int32_t, rhpdhg_result *r) { return fake_poll(++b->polls, r); }
int rhpdhg_batch_remove(rhpdhg_batch *b, int32_t) { b->status = -1; return RHPDHG_OK; }
void rhpdhg_batch_free(rhpdhg_batch *b) { delete b; }
int rhpdhg_create(const rhpdhg_problem *, const rhpdhg_params *, void *, rhpdhg_handle **h) {
  *h = new rhpdhg_handle;
  return RHPDHG_OK;
}
int rhpdhg_solve(rhpdhg_handle *, int) { return RHPDHG_OK; }
int rhpdhg_poll(rhpdhg_handle *h, rhpdhg_result *r) { return fake_poll(++h->polls, r); }
int rhpdhg_cancel(rhpdhg_handle *) { return RHPDHG_OK; }
void rhpdhg_free(rhpdhg_handle *h) { delete h; }
int rhpdhg_params_default(rhpdhg_params *p) { std::memset(p, 0, sizeof(*p)); return RHPDHG_OK; }
}

int main(int argc, char **argv) {
  const int64_t small_nnz = std::atoi(argv[1]);   // 0: the request gets its own handle
  first_rc = std::atoi(argv[2]);
  later_rc = std::atoi(argv[3]);
  rhpdhg_server *s = nullptr;
  if (rhpdhg_server_create(1ll << 30, small_nnz, 2, 8, &s) != RHPDHG_OK) return 1;
  const int64_t rp[2] = {0, 1};
  const int32_t col[1] = {0};
  const double one[1] = {1.0};
  rhpdhg_problem p{};
  p.m_eq = 1; p.n = 1; p.memory = RHPDHG_MEM_HOST; p.nnz = 1;
  p.row_ptr = rp; p.col_idx = col; p.val = p.c = p.rhs = p.l = p.u = one;
  int64_t ticket = 0;
  if (rhpdhg_server_submit(s, &p, nullptr, &ticket) != RHPDHG_OK) return 2;
  double x = -1.0, y = -1.0;
  rhpdhg_result r{};
  r.x = &x;
  r.y = &y;
  int rc = RHPDHG_BUSY;
  for (int i = 0; i < 10000 && rc == RHPDHG_BUSY; ++i) {
    rc = rhpdhg_server_poll(s, ticket, &r, nullptr);
    std::this_thread::sleep_for(std::chrono::milliseconds(1));
  }
  std::printf("%d %d %g %g %g\n", rc, r.status, r.primal_obj, x, y);
  rhpdhg_server_free(s);
  return 0;
}
"""
OK, OOM, CUDA = 0, -2, -3
OPTIMAL, NUMERICAL_ERROR = 1, 6


@pytest.fixture(scope="module")
def program(tmp_path_factory):
    d = tmp_path_factory.mktemp("server")
    src, exe = d / "fakes.cu", d / "server_poll"
    src.write_text(FAKES)
    subprocess.run([_build.nvcc(), *_build.ARCH, *_build.FLAGS, str(src),
                    os.path.join(_build.CSRC, "server.cu"), "-o", str(exe)], check=True)
    return str(exe)


@pytest.mark.parametrize("small_nnz", [10, 0], ids=["batched", "own_handle"])
@pytest.mark.parametrize("first, later, status, x, y", [
    (OK, OK, OPTIMAL, 3.0, 4.0),
    (CUDA, CUDA, NUMERICAL_ERROR, 0.0, 0.0),
], ids=["ok", "cuda_error"])
def test_poll_code_decides_the_status(program, small_nnz, first, later, status, x, y):
    out = subprocess.run([program, str(small_nnz), str(first), str(later)], capture_output=True,
                         text=True, timeout=60, check=True).stdout.split()
    assert int(out[0]) == OK and int(out[1]) == status
    assert [float(v) for v in out[3:]] == [x, y]


def test_batched_slot_out_of_memory_is_polled_again(program):
    out = subprocess.run([program, "10", str(OOM), str(OK)], capture_output=True, text=True,
                         timeout=60, check=True).stdout.split()
    assert [float(v) for v in out] == [OK, OPTIMAL, 7.0, 3.0, 4.0]
