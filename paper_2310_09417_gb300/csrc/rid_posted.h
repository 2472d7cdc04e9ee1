// rid_posted.h -- states that a loop launched ahead of its stop test posts to
// page-locked memory (host code; Rt is the CUDA runtime, or a stand-in on the CPU).
//
// A state is copied in stream order and an event recorded behind it, so that the reader
// waits for that copy alone and not for what was queued after it.  The two slots belong to
// the calling thread and outlive the call, so a call that ends early (an error between a
// post and its read) waits for its copies first: the thread's next call, perhaps on another
// stream, writes the same slots.
#pragma once
#include <stddef.h>
#include <stdint.h>

namespace rid {

template <typename State, typename Rt>
class PostedStates {
 public:
  PostedStates() = default;
  PostedStates(const PostedStates&) = delete;
  PostedStates& operator=(const PostedStates&) = delete;
  ~PostedStates() {
    for (int i = 0; i < 2; ++i) {
      if (pending_[i]) Rt::wait(event_[i]);
      if (made_[i]) Rt::destroy(event_[i]);
    }
  }

  // False when there is no page-locked memory or no event: the caller waits for every state.
  bool open() {
    for (int i = 0; i < 2; ++i)
      if (!made_[i] && !(made_[i] = Rt::create(&event_[i]))) return false;
    return (slots_ = thread_slots()) != nullptr;
  }

  // State number t as of now in `stream`.  At most two are posted and not read.
  bool post(int64_t t, const State* device, typename Rt::Stream stream) {
    const int i = (int)(t & 1);
    if (pending_[i]) Rt::wait(event_[i]);
    pending_[i] = false;
    if (!Rt::copy(&slots_[i], device, sizeof(State), stream)) return false;
    if (!Rt::record(event_[i], stream)) {
      Rt::wait_stream(stream);  // the copy has no event to wait for
      return false;
    }
    return pending_[i] = true;
  }

  bool read(int64_t t, State* out) {
    const int i = (int)(t & 1);
    if (!Rt::wait(event_[i])) return false;
    pending_[i] = false;
    *out = slots_[i];
    return true;
  }

 private:
  // Two slots of the calling thread, freed with it; calls of one thread follow each other.
  static State* thread_slots() {
    struct Holder {
      void* p = nullptr;
      ~Holder() {
        if (p != nullptr) Rt::free_pinned(p);
      }
    };
    static thread_local Holder h;
    if (h.p == nullptr) h.p = Rt::alloc_pinned(2 * sizeof(State));
    return static_cast<State*>(h.p);
  }

  State* slots_ = nullptr;
  typename Rt::Event event_[2] = {};
  bool made_[2] = {false, false}, pending_[2] = {false, false};
};

}  // namespace rid
