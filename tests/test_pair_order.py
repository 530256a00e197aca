"""The issue order of the CTA-pair block kernel (pair_order.h, the code that
the kernel runs) on the host, against modelled barriers whose parity tests
cannot tell a phase from the one two before it: however late a copy or a
softmax step is, every product reads its own block's rows, and no order
stalls. Heads of one block to many, one to nine blocks a cluster."""
import os
import subprocess

from conftest import ROOT


def test_products_wait_for_their_own_blocks(tmp_path):
    exe = str(tmp_path / "pair_order_model")
    subprocess.run(
        ["g++", "-std=c++17", "-O1", "-Wall", "-Wextra", "-Werror",
         "-I", os.path.join(ROOT, "paper_2607_20214_gb300", "csrc"),
         os.path.join(ROOT, "tests", "pair_order_model.cpp"), "-o", exe],
        check=True)
    r = subprocess.run([exe, "240"], capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
