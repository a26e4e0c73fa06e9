// Host side of cs_decode_loop: when a step is sent.  Plain C++, so that it can be run without a device.
#pragma once

// What the device reports after every step in one 64-bit word: (steps done << 32) | the most tokens any
// sequence still has to emit.
struct LoopProgress {
  int steps;
  int wanted;
};
static inline LoopProgress progress_of(unsigned long long word) { return {(int)(word >> 32), (int)(word & 0xffffffffu)}; }

// Looks at the word once.  True when it tells of more steps than *at; both halves are then taken from that one
// look: two looks could pair the tokens of a step with the count of a later one.
template <typename Word>
static inline bool newer_report(Word word, LoopProgress* at) {
  const LoopProgress now = progress_of(word());
  if (now.steps <= at->steps) return false;
  *at = now;
  return true;
}

// Whether the steps in flight will likely be the last: going by the tokens a step has brought so far, they bring all that
// are wanted.  (Certain where a step brings one token.)
static inline bool likely_last(const LoopProgress& at, int sent, int max_new) {
  return at.steps > 0 && (long)at.wanted * at.steps <= (long)(sent - at.steps) * (max_new - at.wanted);
}

// Runs the loop until no sequence wants a token.  At most two steps are ahead of the reports, and a step is sent
// ahead of a report only where it is needed whatever the steps in flight accept (at most k + 1 tokens each).
// `send(n, wanted)` sends step number n (from 1); `wait(&at, sent)` returns with a newer report.  Both return a
// status; the first that is not 0 ends the loop.
template <typename Send, typename Wait>
static inline int drive_loop(int max_new, int k, Send send, Wait wait) {
  LoopProgress at = {0, max_new};
  int sent = 0, status = 0;
  while (status == 0 && at.wanted > 0 && at.steps < max_new) {
    if (sent < max_new && sent - at.steps < 2 && at.wanted > (long)(sent - at.steps) * (k + 1)) {
      ++sent;
      status = send(sent, at.wanted);
    } else {
      status = wait(&at, sent);
    }
  }
  return status;
}
