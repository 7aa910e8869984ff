"""The names under which the binding reports kern_ms and kern_launches stand in the library's order."""
import os
import re

from test_lib_abi import load_builder

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

# the library's enumerators (csrc/host.h) and the binding's names for them
NAMES = dict(K_SKETCH="sketch_gemm", K_LSQR_PASS="lsqr_pass", K_FGM_PASS="fgmres_pass", K_RES_PASS="residual_pass",
             K_ARNOLDI="arnoldi_step", K_TRSV="fgmres_trsv", K_SKETCH_SUM="sketch_sum")


def test_names_follow_the_enumerators():
    load_builder().build()
    import paper_2410_06319_gb300 as lsq
    with open(os.path.join(ROOT, "paper_2410_06319_gb300", "csrc", "host.h")) as fh:
        body = re.search(r"enum Kern \{(.*?)\}", fh.read(), re.S).group(1)
    enums = [e.split("=")[0].strip() for e in body.split(",")]
    assert [NAMES.get(e, "spare7") for e in enums] == lsq.KERNELS, (enums, lsq.KERNELS)
