"""Rules of the kernels' host and device code that need no GPU, compiled into a
small host program from the library's own headers."""

import os
import subprocess

import numpy as np
import pytest

from paper_1507_08751_gb300 import build as B

PROGRAM = r"""
#include <stdio.h>
#include <string.h>
#include "huge.cuh"
using namespace msllr;
int main() {
  char what[16];
  while (scanf("%15s", what) == 1) {
    if (!strcmp(what, "bound")) {
      float thr, g, w;
      int ku;
      if (scanf("%f %f %d %f", &thr, &g, &ku, &w) != 4) return 1;
      printf("%.9g\n", cert_bound(thr, g, ku, w));
    } else if (!strcmp(what, "plan")) {
      int np, B, sms, widest;
      if (scanf("%d %d %d %d", &np, &B, &sms, &widest) != 4) return 1;
      const SubspacePlan p = subspace_plan(np, B, sms, widest);
      printf("%d %d\n", p.cluster, (int)p.phases);
    }
  }
  return 0;
}
"""


@pytest.fixture(scope="module")
def ask(tmp_path_factory):
    d = tmp_path_factory.mktemp("rules")
    src, exe = d / "rules.cu", d / "rules"
    src.write_text(PROGRAM)
    subprocess.run([B.nvcc(), *B.ARCH, "-std=c++17", "-I", B.CSRC, "-o", str(exe), str(src)],
                   check=True, capture_output=True)

    def call(lines):
        out = subprocess.run([str(exe)], input="\n".join(lines), text=True, check=True,
                             capture_output=True).stdout
        return out.split("\n")[:-1]
    return call


@pytest.mark.parametrize("n,ku", [(40, 1), (128, 8), (200, 9), (256, 12), (256, 16)])
def test_certificate_bound_covers_forming_the_deflated_matrix(ask, n, ku):
    """A = G - U What^T - What U^T by 2 ku FP32 multiply-adds an entry: each
    rounds by at most 2^-24 of a partial sum below |G| + 2 |U| |What|^T, so the
    computed A is within 2 ku 2^-24 || |G| + 2 |U| |What|^T ||_2 of the exact one.
    The bound has to leave that room, with |G| given by its trace or its
    largest row sum, whichever is smaller.  (8 (ku + 1) eps of it does not, with
    16 pairs just above a crowd.)"""
    rng = np.random.default_rng(n + ku)
    thr = 1.0
    Q, _ = np.linalg.qr(rng.standard_normal((n, n)))
    for strong in (1.01, 4.0, 36.0):
        for crowd in (0.0, 0.9):
            # every kept pair at the same eigenvalue: the largest ||What||_F for
            # a given norm of G
            lam = np.concatenate([np.full(ku, strong), np.full(n - ku, crowd)])
            G = (Q * lam) @ Q.T
            U = Q[:, :ku]
            W = U * (0.5 * strong)
            T = np.abs(G) + 2.0 * np.abs(U) @ np.abs(W).T
            worst = 2 * ku * 2.0 ** -24 * np.linalg.norm(T, 2)
            gnorm = min(np.trace(G), np.abs(G).sum(axis=1).max())
            c = float(ask([f"bound {thr} {gnorm:.9g} {ku} {(W ** 2).sum():.9g}"])[0])
            # (2^-24: the bound itself is rounded to FP32)
            assert thr - c >= worst - 2.0 ** -24


@pytest.mark.parametrize("blocks", [1, 9, 10, 64])
def test_subspace_plan_needs_sixteen_ctas_above_4096_only(ask, blocks):
    """Every order up to 8192 with clusters of 16, up to 4096 with clusters of 8;
    rows per CTA within the kernels' limits, 16-CTA clusters only where the
    device has them."""
    orders = range(320, 8193, 64)
    for widest in (16, 8):
        got = ask([f"plan {o} {blocks} 152 {widest}" for o in orders])
        assert len(got) == len(orders)
        for o, line in zip(orders, got):
            cluster, phases = (int(v) for v in line.split())
            if widest == 8 and o > 4096:
                assert cluster == 0
                continue
            assert cluster in (8, widest)
            assert o % cluster == 0 and o // cluster <= (512 if phases else 128)
            assert phases == (o > (2048 if widest == 16 else 1024))
            if widest == 16 and blocks < 10:
                assert cluster == (8 if o <= 512 else 16)
