"""What the build leaves in the tree.  No GPU is needed."""
import glob
import os
import sysconfig

from paper_2210_03858_b200 import build as bcq_build


def test_the_extension_carries_the_abi_tag_of_its_interpreter():
    bcq_build.build_library()
    suffix = sysconfig.get_config_var("EXT_SUFFIX")
    assert "cpython" in suffix
    built = glob.glob(os.path.join(bcq_build.HERE, "_bcq_call*.so"))
    assert [os.path.basename(p) for p in built] == ["_bcq_call" + suffix]
