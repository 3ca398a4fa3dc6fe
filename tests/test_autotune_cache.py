"""The tile cache's key: choices timed with other kernels are not reused."""
import hashlib
import json
import shutil

import pytest

pytest.importorskip("torch")

from paper_1408_7069_gb300 import autotune, letkf  # noqa: E402

SHAPES = [(80, 32, 7), (16, 48, 5)]


def test_choices_of_other_kernels_are_timed_again(tmp_path):
    # as the cache was keyed when the wide class still started at 2 x 4
    old = hashlib.sha1(json.dumps(["GPU", 5, sorted(SHAPES)]).encode()).hexdigest()
    assert autotune.signature("GPU", SHAPES) != old
    # any change of the sources gives another revision, the same sources the same one
    a, b = tmp_path / "a", tmp_path / "b"
    for d in (a, b):
        shutil.copytree(letkf.PKG_DIR + "/csrc", d)
    assert autotune.kernel_revision(str(a)) == autotune.kernel_revision(str(b))
    assert autotune.kernel_revision(str(a)) == autotune.kernel_revision()
    autotune.kernel_revision.cache_clear()
    with open(b / "letkf_pair.cu", "a") as f:
        f.write("// another kernel\n")
    assert autotune.kernel_revision(str(a)) != autotune.kernel_revision(str(b))


def test_the_key_depends_on_gpu_and_instances_in_any_order():
    assert autotune.signature("GPU", SHAPES) == autotune.signature("GPU", SHAPES[::-1])
    assert autotune.signature("GPU", SHAPES) != autotune.signature("other", SHAPES)
    assert autotune.signature("GPU", SHAPES) != autotune.signature("GPU", SHAPES[:1])
