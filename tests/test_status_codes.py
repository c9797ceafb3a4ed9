"""Codes that expired waits leave in the device status word, read from the sources."""
import os
import re

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2607_27744_b200", "csrc")


def test_the_claim_of_an_attention_item_has_a_code_of_its_own():
    text = open(os.path.join(CSRC, "umma_dca.cu")).read()
    claim = re.findall(r"claim_cta\([^;]*kStatusDca \| (\d+)\)", text)
    assert len(claim) == 1
    assert len(re.findall(rf"kStatusDca \| {claim[0]}\b|, {claim[0]}\)\)", text)) == 1   # the second form: the producers' wait()
