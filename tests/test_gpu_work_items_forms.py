"""The Krylov launch in the forms that only large sets take, on the work items' small cases: the
1,024-thread instance of a preconditioned FP64 iteration (from 16 million streamed entries on),
and the row loop without a list of work items (a block with more than 768).  The kernel is
compiled with both limits lowered and linked with the library's other objects; the cases and
their bars are test_gpu_work_items.py's.
"""
import importlib
import subprocess

import pytest

from test_gpu_work_items import CASES, test_solves_meet_the_tolerance_in_every_system as check

pytestmark = pytest.mark.gpu

FORMS = {"large": ["-DVIP_LARGE_STREAM=0"], "unlisted": ["-DVIP_ITEM_CAP=3"],
         "large_unlisted": ["-DVIP_LARGE_STREAM=0", "-DVIP_ITEM_CAP=3"]}


@pytest.fixture(scope="module", params=list(FORMS))
def forced(request, vip, tmp_path_factory):
    build = importlib.import_module("paper_1401_6513_gb300.build")
    others = [build.BUILD / (src.stem + ".o") for src in build.sources() if src.stem != "vip_krylov"]
    if not all(o.exists() for o in others):
        build.build(force=True)
    d = tmp_path_factory.mktemp("krylov")
    subprocess.run([build.nvcc(), *build.NVCC_FLAGS, *build.ARCH, "-w", *FORMS[request.param], "-I", str(build.CSRC),
                    "-c", str(build.CSRC / "vip_krylov.cu"), "-o", str(d / "k.o")], check=True)
    subprocess.run([build.nvcc(), *build.ARCH, "-shared", "-o", str(d / "libvip_forced.so"), str(d / "k.o"),
                    *map(str, others), "-lcudart"], check=True)
    usual, vip._lib = vip._lib, vip.lib(d / "libvip_forced.so")
    yield vip
    vip._lib = usual


@pytest.mark.parametrize("form", ["fp64", "mg32", "mixed"])
@pytest.mark.parametrize("name", list(CASES))
def test_forced_form_meets_the_tolerance(forced, name, form):
    check(forced, name, form)
