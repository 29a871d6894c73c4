"""A stored launch shape belongs to the kernels it was timed on: the cache key
follows their source."""
import shutil

from paper_2505_07392_gb300 import igr, inputs


def test_key_follows_the_kernel_source(tmp_path, monkeypatch):
    c = inputs.blast(32)
    key = igr.autotune_key(c, "f16", False, "GB300")
    copy = tmp_path / "package"
    shutil.copytree(igr.HERE + "/csrc", copy / "csrc")
    monkeypatch.setattr(igr, "HERE", str(copy))
    igr._kernel_tag.cache_clear()
    try:
        assert igr.autotune_key(c, "f16", False, "GB300") == key  # the same source elsewhere
        with open(copy / "csrc" / "igr_kernels.cu", "a") as f:
            f.write("// another kernel\n")
        igr._kernel_tag.cache_clear()
        assert igr.autotune_key(c, "f16", False, "GB300") != key
    finally:
        igr._kernel_tag.cache_clear()


def test_a_shape_of_other_kernels_is_not_found(tmp_path):
    """An entry under the key without the kernels (as written before) is left unused."""
    c = inputs.blast(32)
    path = str(tmp_path / "tiles.json")
    key = igr.autotune_key(c, "f16", False, "GB300")
    igr.autotune_cache_store(path, key.split(":kernels")[0], {"tiles": [4, 4, 4], "forms": [0, 0]})
    assert igr.autotune_cache_load(path).get(key) is None
