"""The roofline's headline stage is the longest of all stages, the products and
chirp-z of the alpha sums among them."""
import pytest

from tests.test_bench_roofline_cpu import _Supports, bench  # noqa: F401 (fixture)


class _Plan(_Supports):
    def __init__(self):
        super().__init__(1024, 5, 2.0)
        self.nscale -= 1

    def alpha_method(self, j, direction):
        hi = self.support(j)[1] + 1
        return (0 if hi <= 32 else (2 if hi <= 512 else 1), 0, 0, 0)


@pytest.mark.parametrize("longest", ["syn_alpha_czt+seg", "ana_alpha_czt+seg", "syn_contract", "ana_beta", "syn_alpha_direct"])
def test_dominant_stage_is_the_longest(bench, longest):  # noqa: F811
    ms = {"ana_contract": 0.31, "ana_beta": 0.23, "ana_alpha_czt": 0.2, "ana_alpha_seg": 0.1, "ana_alpha_direct": 0.12,
          "syn_contract": 0.38, "syn_beta": 0.23, "syn_alpha_czt": 0.15, "syn_alpha_seg": 0.15, "syn_alpha_direct": 0.18}
    if longest.endswith("czt+seg"):  # the group's two parts, neither the longest by itself
        ms[longest[:-4]], ms[longest[:4] + "alpha_seg"] = 0.25, 0.25
    else:
        ms[longest] = 0.6
    r = bench.roofline(_Plan(), ms, 2.4)
    assert r["kernel"] == longest and r["timed"] == "stage"
    assert r["ms"] == max(v["ms"] for v in r["kernels"].values())
