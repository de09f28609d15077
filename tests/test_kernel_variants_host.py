"""The kernel-variant harness stays applicable: every variant sets macros that the
current sources leave to the build (no GPU, nothing built)."""
import os
import re

from tests import kernel_variants as K


def test_every_variant_sets_a_macro_of_the_sources():
    src = "".join(open(os.path.join(K.CSRC, f)).read() for f in os.listdir(K.CSRC) if f.endswith((".cu", ".cuh")))
    assert K.VARIANTS
    for family, variants in K.VARIANTS.items():
        assert variants, family
        for name, flags in variants.items():
            macros = [re.fullmatch(r"-D(\w+)(?:\(\w+\))?=\S+", f) for f in flags]
            assert macros and all(macros), (family, name, flags)
            for m in macros:
                guarded = re.search(rf"#ifndef {m[1]}\n#define {m[1]}\b", src)
                used = len(re.findall(rf"\b{m[1]}\b", src)) > 2
                assert guarded and used, f"{family}/{name}: {m[1]} is no macro of the sources"
