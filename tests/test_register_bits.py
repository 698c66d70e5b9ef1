"""The register-bits field of the flags (4 bits): what no kernel has is refused
by every plan entry point, and what is accepted is taken as given."""
import pytest

import synth


@pytest.mark.parametrize("r", range(1, 16))
def test_every_value_of_the_field(r):
    from paper_2205_06973_gb300 import build
    build.build()
    from paper_2205_06973_gb300 import _native as N
    from paper_2205_06973_gb300 import api
    n, t = 14, 10
    plan = api.Plan(synth.layered(n, 4, seed=3), n, "dagp", 8)
    if r > 5:   # 2^(10 - r) threads: less than a warp, or no such kernel
        for call in (lambda: plan.stats("c64", t, regbits=r), lambda: plan.source(0, "c64", t, regbits=r),
                     lambda: plan.specialise("c64", t, load=False, regbits=r),
                     lambda: plan.stats("c64", t, regbits=r, jit=True)):
            with pytest.raises(N.SvError) as e:
                call()
            assert e.value.status == N.SV_ERR_PARTITION
    else:
        assert plan.stats("c64", t, regbits=r)["passes"] > 0
        assert f"__launch_bounds__({1 << (t - r)}," in plan.source(0, "c64", t, regbits=r)
        assert plan.specialise("c64", t, load=False, regbits=r) > 0.0
    plan.close()
