"""Dense model correction (eq. (7)) through lsr_surfel_correct against the
FP64 oracle, on a seeded room-sized surfel map and a keyframe loop with a
drift correction growing to 1.5 deg / 6 cm.

Which keyframes observe a surfel is decided in FP32 on the device and in FP64
in the oracle. The oracle reports the surfels for which some keyframe of their
time window decides visibility within 1e-5 m of a depth limit or 1e-3 pixels of
an image edge (the FP32 transform and projection err by less); only those may
differ. Every other surfel is kept or removed by both, and where kept its
position and normal agree to FP32 rounding (1e-5).
"""
import numpy as np
import pytest

import oracle
from synth.surfels import make_surfels

gpu = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1801_01572_gb300 as lsr
    c = lsr.Context(0)
    yield c
    c.close()


@pytest.fixture(scope="module")
def smap():
    return make_surfels(400_000, 200, seed=9)


@gpu
def test_surfel_correction_matches_oracle(ctx, smap):
    S = smap
    p, n, keep, kept = ctx.surfel_correct(S.pos, S.nrm, S.t0, S.tu, S.T_old, S.T_new, S.t_kf, S.cam)
    pr, nr, keepr, border = oracle.surfel_correct(S.pos, S.nrm, S.t0, S.tu, S.T_old, S.T_new, S.t_kf, S.cam,
                                                  band=(1e-5, 1e-3))
    keep = keep.astype(bool)
    assert kept == keep.sum() and 0.1 < keep.mean() < 0.9
    assert border.mean() < 1e-3
    assert np.array_equal(keep[~border], keepr[~border])
    both = keep & keepr & ~border
    ep = np.linalg.norm(p[both] - pr[both], axis=1)
    en = np.linalg.norm(n[both] - nr[both], axis=1)
    assert ep.max() <= 1e-5 and en.max() <= 1e-5, (ep.max(), en.max())
    assert np.median(ep) < 2e-6
    # removed surfels come back unchanged
    assert np.array_equal(p[~keep], S.pos[~keep]) and np.array_equal(n[~keep], S.nrm[~keep])


@gpu
def test_surfel_correction_device_inputs_equal_host(ctx, smap):
    torch = pytest.importorskip("torch")
    S = smap
    a = ctx.surfel_correct(S.pos, S.nrm, S.t0, S.tu, S.T_old, S.T_new, S.t_kf, S.cam)
    d = [torch.from_numpy(x).cuda() for x in (S.pos, S.nrm, S.t0, S.tu)]
    b = ctx.surfel_correct(*d, S.T_old, S.T_new, S.t_kf, S.cam)
    assert a[3] == b[3]
    for x, y in zip(a[:3], b[:3]):
        assert np.array_equal(x, y.cpu().numpy())


@gpu
def test_surfels_outside_every_window_are_removed_unchanged(ctx, smap):
    S = smap
    n = 1000
    t0 = np.full(n, -10.0, np.float32)
    tu = np.full(n, -5.0, np.float32)  # before the first keyframe
    p, nr, keep, kept = ctx.surfel_correct(S.pos[:n], S.nrm[:n], t0, tu, S.T_old, S.T_new, S.t_kf, S.cam)
    assert kept == 0 and not keep.any()
    assert np.array_equal(p, S.pos[:n]) and np.array_equal(nr, S.nrm[:n])


@gpu
@pytest.mark.parametrize("n", [1, 31, 512, 513, 2051, 470_001])
@pytest.mark.parametrize("m", [1, 2, 300, 600])
def test_small_keyframe_tables_equal_the_general_kernel(ctx, n, m):
    """A table of up to 600 keyframes takes the tile kernel. Keyframes stamped
    after every surfel's window change nothing, but 601 and more rows take the
    general kernel: the same bits, with surfels of empty windows among them."""
    S = make_surfels(n, m, seed=31 + m)
    t0, tu = S.t0.copy(), S.tu.copy()
    tu[::7] = t0[::7]          # empty windows
    t0[::11], tu[::11] = -5.0, 1e6
    extra = 601
    far = np.tile(np.eye(4), (extra, 1, 1))
    a = ctx.surfel_correct(S.pos, S.nrm, t0, tu, S.T_old, S.T_new, S.t_kf, S.cam)
    b = ctx.surfel_correct(S.pos, S.nrm, t0, tu, np.concatenate([S.T_old, far]), np.concatenate([S.T_new, far]),
                           np.concatenate([S.t_kf, 2e6 + np.arange(extra, dtype=np.float32)]), S.cam)
    assert a[3] == b[3]
    for x, y in zip(a[:3], b[:3]):
        assert np.array_equal(x, y)


_THREADS_C = r"""
#include <pthread.h>
#include <stdio.h>
#include <stdlib.h>

#include "lsr.h"

enum { kThreads = 8, kSurfels = 64, kCalls = 3000 };

/* A context of its own and a table of 600 or of 1 keyframes; returns the calls that failed. */
static void *work(void *arg) {
  const int m = (long)arg % 2 ? 600 : 1;
  lsr_ctx *ctx = NULL;
  if (lsr_create(&ctx, NULL, 0, NULL) != LSR_OK) return (void *)(long)kCalls;
  float *pos = calloc(3 * kSurfels, 4), *nrm = calloc(3 * kSurfels, 4), *t0 = calloc(kSurfels, 4);
  float *tu = calloc(kSurfels, 4), *po = calloc(3 * kSurfels, 4), *no = calloc(3 * kSurfels, 4);
  uint8_t *keep = calloc(kSurfels, 1);
  double *T = calloc(16 * (size_t)m, 8);
  float *tk = calloc(m, 4);
  const float cam[7] = {500, 500, 320, 240, 640, 480, 5};
  for (int f = 0; f < m; ++f) {
    for (int k = 0; k < 16; k += 5) T[16 * f + k] = 1;
    tk[f] = (float)(f + 1);
  }
  for (int i = 0; i < kSurfels; ++i) pos[3 * i + 2] = nrm[3 * i + 2] = 1, tu[i] = 1e6f;
  long bad = 0;
  for (int c = 0; c < kCalls; ++c) {
    int64_t kept = 0;
    const int rc = lsr_surfel_correct(ctx, kSurfels, pos, nrm, t0, tu, m, T, T, tk, cam, po, no, keep, &kept);
    bad += rc != LSR_OK || kept != kSurfels;
  }
  lsr_destroy(ctx);
  return (void *)bad;
}

int main(void) {
  pthread_t t[kThreads];
  long bad = 0;
  for (long k = 0; k < kThreads; ++k) pthread_create(t + k, NULL, work, (void *)k);
  for (int k = 0; k < kThreads; ++k) {
    void *r;
    pthread_join(t[k], &r);
    bad += (long)r;
  }
  printf("%ld\n", bad);
  return 0;
}
"""


@gpu
def test_threads_with_tables_of_different_sizes(tmp_path):
    """Contexts on eight threads, half with 600 keyframes and half with one:
    the kernel's limit of shared memory is the device's, not the call's, so no
    call may narrow it between another's setting and launch. Every call
    succeeds. (In C: with an interpreter between the calls hardly any meet.)"""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import os
    import subprocess

    from paper_1801_01572_gb300 import _build
    src, exe = tmp_path / "threads.c", tmp_path / "threads"
    src.write_text(_THREADS_C)
    subprocess.run(["gcc", "-O1", "-I", os.path.join(_build.ROOT, "include"), str(src), _build.LIB, "-o", str(exe),
                    "-lpthread", "-Wl,-rpath," + _build.OUT], check=True)
    out = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120, check=True)
    assert int(out.stdout) == 0
