// idle_list.h -- the bookkeeping of a bounded list of idle objects that belong
// to owners which may have gone (plans.cu); host only, no CUDA.
#pragma once

namespace flame {

// At most Most idle objects, oldest first.  Key has operator== and `ctx`, the
// owner: an object may be destroyed only while its owner is there, which is known
// of the caller's owner alone.
template <class Key, class Object, int Most>
class IdleList {
 public:
  // Takes out the youngest object of this key; false if there is none.
  bool take(const Key& k, Object* o) {
    for (int i = n_ - 1; i >= 0; --i)
      if (key_[i] == k) {
        *o = remove(i);
        return true;
      }
    return false;
  }
  // Keeps o.  True if *drop has to be destroyed, by k's owner, which has it: the
  // oldest object of the same owner where the list is full, or o itself where the
  // list is full of others' objects.
  bool give(const Key& k, Object o, Object* drop) {
    bool full = n_ == Most;
    if (full) {
      *drop = o;
      for (int i = 0; i < n_; ++i)
        if (key_[i].ctx == k.ctx) {
          *drop = remove(i);
          break;
        }
      if (n_ == Most) return true;
    }
    key_[n_] = k;
    object_[n_++] = o;
    return full;
  }
  int size() const { return n_; }

 private:
  Object remove(int i) {
    const Object o = object_[i];
    --n_;
    for (int j = i; j < n_; ++j) {
      key_[j] = key_[j + 1];
      object_[j] = object_[j + 1];
    }
    return o;
  }
  Key key_[Most];
  Object object_[Most];
  int n_ = 0;
};

}  // namespace flame
